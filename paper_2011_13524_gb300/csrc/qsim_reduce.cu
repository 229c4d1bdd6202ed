// Reductions over a state vector (Sec. 4.2.2 squared norm and inner product, Sec. 4.5
// Pauli-observable expectation and transition amplitude) and the out-of-place product
// lambda = O psi used by the adjoint gradient.
//
// Sums are deterministic: every block writes its partial sums to its own slot, and one
// block adds the slots in a fixed order. Accumulation is FP64 for both storage types;
// complex64 amplitudes are widened to double before they are multiplied.
//
// Expectation: the terms of O = sum_P alpha_P P are grouped by their flip mask f (the
// X-or-Y positions). Group f = 0 is diagonal: sum_y w(y) |psi_y|^2 with
// w(y) = sum_P alpha_P (-1)^{popcount(y & z_P)}. A group f != 0 visits each pair
// (y, y ^ f) once, with A = conj(psi_{y^f}) psi_y:
//   <psi|P|psi> restricted to the pair = i^{#Y} (s(y) A + s(y^f) conj(A)).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <mutex>
#include <type_traits>

#include "qsim_arith.cuh"

namespace qs {

namespace {

constexpr int kRedThreads = 256;
constexpr int kMaxTermsPerLaunch = 48;
static_assert(kHeavyChunkTerms <= kMaxTermsPerLaunch, "heavy chunks must fit one launch");

int sms() { return device_sms(); }

unsigned red_grid(uint64_t work) {
    const uint64_t want = (work + kRedThreads * 4 - 1) / (kRedThreads * 4);
    return unsigned(std::max<uint64_t>(1, std::min<uint64_t>(want, uint64_t(sms()) * 4)));
}

// Block partial of (re, im) pairs into part[2*blockIdx.x + {0,1}].
__device__ __forceinline__ void write_partial2(double re, double im, double* part) {
    __shared__ double sh[kRedThreads / 32];
    const double r = block_sum<kRedThreads>(re, sh);
    const double i = block_sum<kRedThreads>(im, sh);
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = r;
        part[2 * blockIdx.x + 1] = i;
    }
}

template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_norm2(const C* __restrict__ psi, uint64_t N, double* part) {
    double acc = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t x = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < N; x += stride) {
        const double2 v = widen(psi[x]);
        acc = fma(v.x, v.x, acc);
        acc = fma(v.y, v.y, acc);
    }
    write_partial2(acc, 0.0, part);
}

template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_inner(const C* __restrict__ a, const C* __restrict__ b, uint64_t N,
                                                       double* part) {
    double re = 0.0, im = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t x = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; x < N; x += stride) {
        const double2 u = widen(a[x]), v = widen(b[x]);
        re = fma(u.x, v.x, re);
        re = fma(u.y, v.y, re);
        im = fma(u.x, v.y, im);
        im = fma(-u.y, v.x, im);
    }
    write_partial2(re, im, part);
}

struct TermParams {
    uint64_t xmask;          // group flip mask
    IndexPlan ip;            // pivot bit inserted (f != 0) or plain range (f == 0)
    int32_t nterms;
    double coef[kMaxTermsPerLaunch];
    uint64_t zmask[kMaxTermsPerLaunch];
    int32_t nY[kMaxTermsPerLaunch];
};

template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_expect_group(const C* __restrict__ psi,
                                                              const __grid_constant__ TermParams P, double* part) {
    double re = 0.0, im = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < P.ip.n_iter; i += stride) {
        const uint64_t y = expand(i, P.ip);
        if (P.xmask == 0) {
            const double2 v = widen(psi[y]);
            const double p = fma(v.x, v.x, v.y * v.y);
            double w = 0.0;
            for (int t = 0; t < P.nterms; t++) w += parity64(y & P.zmask[t]) ? -P.coef[t] : P.coef[t];
            re = fma(w, p, re);
        } else {
            const uint64_t y2 = y ^ P.xmask;
            const double2 a = widen(psi[y]), b = widen(psi[y2]);
            const double Ar = fma(b.x, a.x, b.y * a.y);   // A = conj(b) a
            const double Ai = fma(b.x, a.y, -b.y * a.x);
            for (int t = 0; t < P.nterms; t++) {
                const int s1 = parity64(y & P.zmask[t]);
                const int s2 = parity64(y2 & P.zmask[t]);
                // s1 A + s2 conj(A): equal signs -> 2 s Re A ; opposite -> 2 i s Im A
                double ur, ui;
                const double sg = s1 ? -2.0 : 2.0;
                if (s1 == s2) { ur = sg * Ar; ui = 0.0; } else { ur = 0.0; ui = sg * Ai; }
                double vr, vi;  // multiply by i^{nY}
                switch (P.nY[t] & 3) {
                    case 0: vr = ur; vi = ui; break;
                    case 1: vr = -ui; vi = ur; break;
                    case 2: vr = -ur; vi = -ui; break;
                    default: vr = ui; vi = -ur; break;
                }
                re = fma(P.coef[t], vr, re);
                im = fma(P.coef[t], vi, im);
            }
        }
    }
    write_partial2(re, im, part);
}

// One term per flip group (general Pauli strings): sum over the pairs (y, y ^ f) of
// (-1)^popc(y & z) Re A or Im A with A = conj(psi_{y^f}) psi_y, whichever the string takes, many terms
// in one launch (blockIdx.y). The coefficient and the pair's factor enter once per block.
//  * complex128: two FP64 FMA per pair, the FP64 rate being the bound (the group kernel below takes
//    seven per pair and term).
//  * complex64: products exact in FP32 pairs, summed with two levels of compensation (TwoSum of the
//    sums and of their errors: nothing above 2^-70 of a thread's sum is dropped), both components of a
//    pair side by side in packed instructions; one FP64 conversion per thread. Where a product
//    lies below 2^-100 (its rounding error can fall under FP32's range) or from 2^80 on, the four pairs
//    loaded with it go to an FP64 sum instead, as the group kernel forms it.
// 24 random strings, whole call, one launch per group / here: complex64 1.62 / 0.36 ms at n = 23 (300 us
// of kernel, 15 of them for the range; L2 reads and packed FP32 arithmetic about equal) and 67.8 / 9.4 ms
// at n = 28, complex128 0.75 / 0.37 ms at n = 22 and 50.9 / 17.9 ms at n = 28.
constexpr int kMaxSingles = 64;
struct SingleTerm {
    uint64_t f, z;
    double coef;     // with the pair's factor +-2
    int32_t pivot;   // highest bit of f, clear in y: runs of y and y ^ f then fill their lines (a string that
                     // flips qubits 0 and 25 at n = 26, complex128: 0.37 ms from the lowest bit, 0.24 from the highest)
    int32_t imag;    // 1: Im A
};
struct SingleParams {
    uint64_t pairs;
    SingleTerm t[kMaxSingles];
};

__device__ __forceinline__ float2 two_sum2(float2 a, float2 b, float2& e) {
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 h = __fadd2_rn(a, b);
    const float2 bp = __ffma2_rn(a, m1, h);
    e = __fadd2_rn(__ffma2_rn(__ffma2_rn(bp, m1, h), m1, a), __ffma2_rn(bp, m1, b));
    return h;
}
struct SingleAccF {  // complex64
    float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f), d = make_float2(0.f, 0.f);
    double wide = 0.0;
    // at least kRange for a product outside [2^-100, 2^80), zero included (the shift drops the sign)
    static constexpr uint32_t kRange = 180u << 24;
    __device__ __forceinline__ static uint32_t range(float p) { return 2u * __float_as_uint(p) - (27u << 24); }
    // the factors of a pair's two products
    __device__ __forceinline__ static float2 factor(float2 a, bool imag, int neg) {
        const uint32_t sg = uint32_t(neg) << 31;
        const float2 u = imag ? make_float2(a.y, -a.x) : a;
        return make_float2(__uint_as_float(__float_as_uint(u.x) ^ sg), __uint_as_float(__float_as_uint(u.y) ^ sg));
    }
    __device__ __forceinline__ static bool in_range(float2 a, float2 b, bool imag, int neg) {
        const float2 p = __fmul2_rn(factor(a, imag, neg), b);
        return max(range(p.x), range(p.y)) < kRange;
    }
    // the same, or a product that a factor makes zero, which is exact (real and sparse states: 24 strings at
    // n = 28 10.8 ms, general ones 9.4, amplitudes spread over 97 binary orders 36, per group 75)
    __device__ __forceinline__ static bool in_range_or_zero(float2 a, float2 b, bool imag, int neg) {
        const float2 u = factor(a, imag, neg), p = __fmul2_rn(u, b);
        return (range(p.x) < kRange || u.x == 0.f || b.x == 0.f) && (range(p.y) < kRange || u.y == 0.f || b.y == 0.f);
    }
    __device__ __forceinline__ void add_wide(float2 a, float2 b, bool imag, int neg) {
        const float2 u = factor(a, imag, neg);
        wide = fma(widen_float_int(u.x), widen_float_int(b.x), wide);
        wide = fma(widen_float_int(u.y), widen_float_int(b.y), wide);
    }
    __device__ __forceinline__ void add(float2 a, float2 b, bool imag, int neg) {
        const float2 u = factor(a, imag, neg), p = __fmul2_rn(u, b);
        float2 e, e2;
        s = two_sum2(s, p, e);
        e = __fadd2_rn(e, __ffma2_rn(u, b, make_float2(-p.x, -p.y)));
        c = two_sum2(c, e, e2);
        d = __fadd2_rn(d, e2);
    }
    __device__ double value() const {
        return ((double(s.x) + double(s.y)) + ((double(c.x) + double(c.y)) + (double(d.x) + double(d.y)))) + wide;
    }
};
struct SingleAccD {  // complex128
    double s = 0.0, c = 0.0;
    __device__ __forceinline__ static bool in_range(double2, double2, bool, int) { return true; }
    __device__ __forceinline__ static bool in_range_or_zero(double2, double2, bool, int) { return true; }
    __device__ __forceinline__ void add(double2 a, double2 b, bool imag, int neg) {
        const long long sg = static_cast<long long>(uint64_t(neg) << 63);
        const double ux = imag ? a.y : a.x, uy = imag ? -a.x : a.y;
        s = fma(__longlong_as_double(__double_as_longlong(ux) ^ sg), b.x, s);
        c = fma(__longlong_as_double(__double_as_longlong(uy) ^ sg), b.y, c);
    }
    __device__ __forceinline__ void add_wide(double2 a, double2 b, bool imag, int neg) { add(a, b, imag, neg); }
    __device__ double value() const { return s + c; }
};

template <typename C, typename Acc>
__global__ void __launch_bounds__(kRedThreads) k_expect_singles(const C* __restrict__ psi,
                                                                const __grid_constant__ SingleParams P, double* part) {
    const SingleTerm T = P.t[blockIdx.y];
    const uint64_t lowmask = (1ull << T.pivot) - 1ull;
    const bool imag = T.imag != 0;
    Acc acc;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    constexpr int kU = 4;  // pairs in flight per thread
    for (uint64_t i0 = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i0 < P.pairs; i0 += kU * stride) {
        C a[kU], b[kU];
        int neg[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) {
            const uint64_t i = i0 + u * stride;
            if (i >= P.pairs) break;
            const uint64_t lo = i & lowmask, y = ((i ^ lo) << 1) | lo;
            a[u] = psi[y];
            b[u] = psi[y ^ T.f];
            neg[u] = parity64(y & T.z);
        }
        const bool four = i0 + (kU - 1) * stride < P.pairs;
        bool fast = four;  // (one branch for the four: their sums interleave)
        if (four) {
#pragma unroll
            for (int u = 0; u < kU; u++) fast &= Acc::in_range(a[u], b[u], imag, neg[u]);
            if (!fast) {  // real or sparse states
                fast = true;
#pragma unroll
                for (int u = 0; u < kU; u++) fast &= Acc::in_range_or_zero(a[u], b[u], imag, neg[u]);
            }
        }
        if (fast) {
#pragma unroll
            for (int u = 0; u < kU; u++) acc.add(a[u], b[u], imag, neg[u]);
        } else {
#pragma unroll
            for (int u = 0; u < kU; u++) {
                if (i0 + u * stride >= P.pairs) break;
                acc.add_wide(a[u], b[u], imag, neg[u]);
            }
        }
    }
    __shared__ double sh[kRedThreads / 32];
    const double r = block_sum<kRedThreads>(acc.value(), sh);
    if (threadIdx.x == 0) {
        const size_t slot = size_t(blockIdx.y) * gridDim.x + blockIdx.x;
        part[2 * slot] = T.coef * r;
        part[2 * slot + 1] = 0.0;
    }
}

// <lam| P |psi> = sum_y conj(lam_y) i^{#Y} s(y ^ f) psi_{y ^ f}
template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_transition(const C* __restrict__ lam, const C* __restrict__ psi,
                                                            uint64_t N, uint64_t xmask, uint64_t zmask, int nY,
                                                            double* part) {
    double re = 0.0, im = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t y = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; y < N; y += stride) {
        const uint64_t y2 = y ^ xmask;
        const double2 l = widen(lam[y]);
        double2 p = widen(psi[y2]);
        p = mul_ipow(p, nY + 2 * parity64(y2 & zmask));
        re = fma(l.x, p.x, re);
        re = fma(l.y, p.y, re);
        im = fma(l.x, p.y, im);
        im = fma(-l.y, p.x, im);
    }
    write_partial2(re, im, part);
}

// <bra| sum_t coef_t P_t |ket> over the terms of one flip group: sum_y conj(bra_y) coef_t i^nY_t
// (-1)^popc(x & z_t) ket_x with x = y ^ xmask (P_t |x> lands on |y>)
template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_transition_group(const C* __restrict__ bra, const C* __restrict__ ket,
                                                                  uint64_t N, const __grid_constant__ TermParams P,
                                                                  double* part) {
    double re = 0.0, im = 0.0;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t y = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; y < N; y += stride) {
        const uint64_t x = y ^ P.xmask;
        const double2 b = widen(bra[y]), k = widen(ket[x]);
        const double vr = fma(b.x, k.x, b.y * k.y), vi = fma(b.x, k.y, -b.y * k.x);  // conj(b) k
        for (int t = 0; t < P.nterms; t++) {
            const double w = parity64(x & P.zmask[t]) ? -P.coef[t] : P.coef[t];
            const double ur = w * vr, ui = w * vi;
            switch (P.nY[t] & 3) {
                case 0: re += ur; im += ui; break;
                case 1: re -= ui; im += ur; break;
                case 2: re -= ur; im -= ui; break;
                default: re += ui; im -= ur; break;
            }
        }
    }
    write_partial2(re, im, part);
}

// sum of |psi_x|^2 over the x whose measured bits are fixed: i runs over the free qubits in
// ascending order, the measured bits set from `set`. x is formed from i by the shorter of two
// loops, the same x either way: one free bit deposited per step, or a zero inserted at each
// measured position (ascending). At n = 28 with 4 measured qubits (24 free): 201 us with 24
// deposits per amplitude, 155 us with 4 insertions (four loads in
// flight per thread measured no faster).
struct FreeBits {
    uint64_t set;
    int32_t nfree, nfix;
    int32_t insert;  // 1: pos holds the measured positions, 0: the free ones
    int8_t pos[64];
};
template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_norm2_sub(const C* __restrict__ psi, const __grid_constant__ FreeBits F,
                                                           double* part) {
    double acc = 0.0;
    const uint64_t n_iter = 1ull << F.nfree;
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n_iter; i += stride) {
        uint64_t x = F.set;
        if (F.insert) {
            uint64_t y = i;
#pragma unroll 1
            for (int j = 0; j < F.nfix; j++) {
                const uint64_t lo = y & ((1ull << F.pos[j]) - 1ull);
                y = ((y ^ lo) << 1) | lo;
            }
            x |= y;
        } else {
#pragma unroll 1
            for (int j = 0; j < F.nfree; j++) x |= ((i >> j) & 1ull) << F.pos[j];
        }
        const double2 v = widen(psi[x]);
        acc = fma(v.x, v.x, acc);
        acc = fma(v.y, v.y, acc);
    }
    write_partial2(acc, 0.0, part);
}

// |v|^2 of an amplitude as an unevaluated FP32 pair (2^-45 relative): the parts split on the integer
// pipes, exact hi x hi products
__device__ __forceinline__ void df_square_sum(float xh, float xl, float yh, float yl, float& s, float& c) {
    const float p = __fmul_rn(xh, xh), q = __fmul_rn(yh, yh);
    const float e = __fmaf_rn(__fadd_rn(xh, xh), xl, __fmaf_rn(xh, xh, -p));
    const float f = __fmaf_rn(__fadd_rn(yh, yh), yl, __fmaf_rn(yh, yh, -q));
    float t;
    DFArith::two_sum(p, q, s, t);
    c = __fadd_rn(t, __fadd_rn(e, f));
}
__device__ __forceinline__ void df_mass(double2 v, float& s, float& c) {
    float xh, xl, yh, yl;
    split_double_int(v.x, xh, xl);
    split_double_int(v.y, yh, yl);
    df_square_sum(xh, xl, yh, yl, s, c);
}
__device__ __forceinline__ void df_mass(float2 v, float& s, float& c) { df_square_sum(v.x, 0.f, v.y, 0.f, s, c); }
__device__ __forceinline__ void df_mass(float4 v, float& s, float& c) { df_square_sum(v.x, v.y, v.z, v.w, s, c); }
// (s, c) += (os, oc)
__device__ __forceinline__ void df_pair_add(float& s, float& c, float os, float oc) {
    float h, e;
    DFArith::two_sum(s, os, h, e);
    s = h;
    c = __fadd_rn(c, __fadd_rn(oc, e));
}

constexpr int kSampleChunkLog = 12;                       // amplitudes per sampling chunk
constexpr int kSegsPerChunk = (1 << kSampleChunkLog) / 32;  // segments of 32 amplitudes

// sampling, step 1: probability mass of each chunk of 2^chunk_log amplitudes (one block each).
// kSegs (chunks of 2^12): also the mass of every 32-amplitude segment as an FP32 pair, for
// k_sample_pick. The FP64 chunk mass bounds the kernel (two FMA per amplitude, GB300's FP64 rate),
// the segment sums run on the idle FP32 and integer pipes beside it: 1060 us without
// them at n = 28 (complex128), 1441 us with them.
template <typename C, bool kSegs>
__global__ void __launch_bounds__(kRedThreads) k_chunk_mass(const C* __restrict__ psi, uint64_t N, int chunk_log,
                                                            double* mass, float2* __restrict__ segs) {
    const uint64_t base = uint64_t(blockIdx.x) << chunk_log;
    if constexpr (kSegs) {
        constexpr int J = (1 << kSampleChunkLog) / kRedThreads;  // amplitudes per thread
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        C v[J];
#pragma unroll
        for (int j = 0; j < J; j++) v[j] = psi[base + threadIdx.x + j * kRedThreads];
        double acc = 0.0;
        float s[J], c[J];
#pragma unroll
        for (int j = 0; j < J; j++) {
            const double2 w = widen(v[j]);
            acc = fma(w.x, w.x, acc);
            acc = fma(w.y, w.y, acc);
            df_mass(v[j], s[j], c[j]);
        }
        // J sums over the warp's lanes at once: in each of the first four stages a lane keeps half of
        // its sums and gives the other half away, so lane l ends with segment j(l)'s sum over 16
        // lanes, and a last stage adds the two halves
        int own = 0;
#pragma unroll
        for (int half = J / 2, bit = 1; half >= 1; half /= 2, bit <<= 1) {
            const bool up = (lane & bit) != 0;
            own = own * 2 + (up ? 1 : 0);
#pragma unroll
            for (int j = 0; j < half; j++) {
                const float gs = up ? s[j] : s[j + half], gc = up ? c[j] : c[j + half];
                if (up) {
                    s[j] = s[j + half];
                    c[j] = c[j + half];
                }
                df_pair_add(s[j], c[j], __shfl_xor_sync(0xffffffffu, gs, bit), __shfl_xor_sync(0xffffffffu, gc, bit));
            }
        }
        df_pair_add(s[0], c[0], __shfl_xor_sync(0xffffffffu, s[0], 16), __shfl_xor_sync(0xffffffffu, c[0], 16));
        // segment (j, warp) covers amplitudes j * 256 + warp * 32 ..
        if (lane < 16) segs[size_t(blockIdx.x) * kSegsPerChunk + own * (kRedThreads / 32) + warp] = make_float2(s[0], c[0]);
        __shared__ double sh[kRedThreads / 32];
        const double r = block_sum<kRedThreads>(acc, sh);
        if (threadIdx.x == 0) mass[blockIdx.x] = r;
        return;
    }
    const uint64_t end = N < base + (1ull << chunk_log) ? N : base + (1ull << chunk_log);
    double acc = 0.0;
    for (uint64_t x = base + threadIdx.x; x < end; x += blockDim.x) {
        const double2 v = widen(psi[x]);
        acc = fma(v.x, v.x, acc);
        acc = fma(v.y, v.y, acc);
    }
    __shared__ double sh[kRedThreads / 32];
    const double r = block_sum<kRedThreads>(acc, sh);
    if (threadIdx.x == 0) mass[blockIdx.x] = r;
}

// sampling, step 2: each sample's chunk (the first whose cumulative mass exceeds u * total; at the
// top, where rounding may leave none, the last chunk with mass) and residual target
__global__ void __launch_bounds__(kRedThreads) k_sample_chunk(const double* __restrict__ cum, uint64_t B,
                                                              const double* __restrict__ u, double total,
                                                              uint64_t last, int count, uint64_t* __restrict__ chunk,
                                                              double* __restrict__ resid) {
    const int k = int(blockIdx.x * blockDim.x + threadIdx.x);
    if (k >= count) return;
    const double target = __dmul_rn(u[k], total);
    uint64_t lo = 0, hi = B;  // first c in [0, B) with cum[c + 1] > target, B if none
    while (lo < hi) {
        const uint64_t mid = (lo + hi) >> 1;
        if (cum[mid + 1] > target) hi = mid; else lo = mid + 1;
    }
    const uint64_t c = lo < B ? lo : last;
    chunk[k] = c;
    resid[k] = __dsub_rn(target, cum[c]);
}

// sampling, step 3: one warp finds, inside the sample's chunk, the first x whose running mass
// (lanes own consecutive stretches, summed in order, FP64) exceeds the residual target
template <typename C>
__device__ __forceinline__ void sample_find_warp(const C* __restrict__ psi, uint64_t N, int chunk_log, uint64_t base,
                                                 double r, int lane, uint64_t* __restrict__ out) {
    const uint64_t len = N - base < (1ull << chunk_log) ? N - base : (1ull << chunk_log);
    const uint64_t per = (len + 31) / 32;
    const uint64_t lo = len < uint64_t(lane) * per ? len : uint64_t(lane) * per;
    const uint64_t hi = len < lo + per ? len : lo + per;
    auto mass = [&](uint64_t x) {
        const double2 v = widen(psi[base + x]);
        return fma(v.x, v.x, v.y * v.y);
    };
    double own = 0.0;
    for (uint64_t x = lo; x < hi; x++) own += mass(x);
    double incl = own;  // inclusive scan over lanes, in lane order
    for (int d = 1; d < 32; d <<= 1) {
        const double v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
    }
    const unsigned over = __ballot_sync(0xffffffffu, incl > r);
    const unsigned nonzero = __ballot_sync(0xffffffffu, own > 0.0);
    // the lane whose stretch crosses r; past the end (rounding) the last lane with mass
    const int L = over ? __ffs(over) - 1 : (nonzero ? 31 - __clz(nonzero) : 31);
    if (lane == L) {
        double acc = incl - own;
        uint64_t pick = hi > lo ? hi - 1 : lo, last = pick;
        bool found = false;
        for (uint64_t x = lo; x < hi; x++) {
            const double m = mass(x);
            if (m > 0.0) last = x;
            acc += m;
            if (acc > r) {
                pick = x;
                found = true;
                break;
            }
        }
        *out = base + (found ? pick : last);
    }
}
template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_sample_find(const C* __restrict__ psi, uint64_t N, int chunk_log,
                                                             const uint64_t* __restrict__ chunk,
                                                             const double* __restrict__ resid, int count,
                                                             uint64_t* __restrict__ out) {
    const int s = int((uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5);
    if (s >= count) return;
    sample_find_warp(psi, N, chunk_log, chunk[s] << chunk_log, resid[s], threadIdx.x & 31, out + s);
}

// The same from the segment masses: the segment by a scan of the chunk's 128 segment sums (FP32
// pairs, four per lane), then the amplitude by a scan of the segment's 32 masses: 1.5 KB read per
// sample instead of the chunk's 64 KB (complex128), and no FP64. The pick stands only where r lies
// further than 2^-38 of the chunk's mass from both of its edges, which is beyond what the FP64 sums
// of k_sample_find (under 2^-44) and the pairs here (under 2^-40) can be off, so both kernels return
// the same index; any other sample (about 1 in 2^25, and every one of a chunk whose mass leaves the
// range where FP32 pairs hold it) is found as there. 10^5 samples at n = 28: 4254 us by the
// chunk search, 91 us here.
template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_sample_pick(const C* __restrict__ psi, uint64_t N,
                                                             const uint64_t* __restrict__ chunk,
                                                             const double* __restrict__ resid,
                                                             const float2* __restrict__ segs, int count,
                                                             uint64_t* __restrict__ out) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int k = int((uint64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5);
    if (k >= count) return;
    const uint64_t ch = chunk[k], base = ch << kSampleChunkLog;
    const double r = resid[k];
    float rh, rl;
    split_double(r, rh, rl);
    auto scan = [&](float& s, float& c) {  // inclusive over the lanes
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float os = __shfl_up_sync(kAll, s, d), oc = __shfl_up_sync(kAll, c, d);
            if (lane >= d) df_pair_add(s, c, os, oc);
        }
    };
    auto above = [&](float s, float c) { return __fadd_rn(__fsub_rn(s, rh), __fsub_rn(c, rl)); };  // (s + c) - r
    constexpr int kPer = kSegsPerChunk / 32;
    float s[kPer], c[kPer];
#pragma unroll
    for (int j = 0; j < kPer; j++) {
        const float2 v = segs[ch * kSegsPerChunk + lane * kPer + j];
        s[j] = v.x;
        c[j] = v.y;
        if (j) df_pair_add(s[j], c[j], s[j - 1], c[j - 1]);
    }
    float ts = s[kPer - 1], tc = c[kPer - 1];
    scan(ts, tc);
    const float total = __shfl_sync(kAll, ts, 31);
    float es = __shfl_up_sync(kAll, ts, 1), ec = __shfl_up_sync(kAll, tc, 1);  // exclusive
    if (lane == 0) es = ec = 0.f;
    bool fine = total > 0x1p-60f && total < 0x1p60f && r >= 0.0;
    // first segment whose inclusive sum exceeds r
    int j = kPer;
    float ps = es, pc = ec;  // its exclusive sum
#pragma unroll
    for (int i = kPer - 1; i >= 0; i--) {
        float is = s[i], ic = c[i];
        df_pair_add(is, ic, es, ec);
        if (above(is, ic) > 0.f) j = i;
    }
#pragma unroll
    for (int i = 0; i < kPer - 1; i++)
        if (j == i + 1) {
            ps = s[i];
            pc = c[i];
            df_pair_add(ps, pc, es, ec);
        }
    const unsigned over = __ballot_sync(kAll, j < kPer);
    fine = fine && over != 0u;
    const int L = over ? __ffs(over) - 1 : 0;
    const int seg = L * kPer + min(__shfl_sync(kAll, j, L), kPer - 1);
    ps = __shfl_sync(kAll, ps, L);
    pc = __shfl_sync(kAll, pc, L);
    // first amplitude of the segment whose inclusive sum exceeds r
    const uint64_t x = base + uint64_t(seg) * 32 + lane;
    float ms, mc;
    df_mass(psi[x], ms, mc);
    scan(ms, mc);
    df_pair_add(ms, mc, ps, pc);
    float bs = __shfl_up_sync(kAll, ms, 1), bc = __shfl_up_sync(kAll, mc, 1);
    if (lane == 0) {
        bs = ps;
        bc = pc;
    }
    const unsigned hit = __ballot_sync(kAll, above(ms, mc) > 0.f);
    const int lx = hit ? __ffs(hit) - 1 : 0;
    const float margin = total * 0x1p-38f;
    const bool clear = lane != lx || (above(ms, mc) > margin && above(bs, bc) < -margin);
    fine = fine && hit != 0u && __all_sync(kAll, clear);
    if (fine) {
        if (lane == lx) out[k] = x;
        return;
    }
    sample_find_warp(psi, N, kSampleChunkLog, base, r, lane, out + k);
}

// sum of `nslots` (re, im) partials in a fixed order -> out[0..1]
__global__ void __launch_bounds__(kRedThreads) k_final2(const double* __restrict__ part, int nslots, double* out) {
    __shared__ double sh[kRedThreads / 32];
    double re = 0.0, im = 0.0;
    for (int j = threadIdx.x; j < nslots; j += kRedThreads) {
        re += part[2 * j];
        im += part[2 * j + 1];
    }
    const double r = block_sum<kRedThreads>(re, sh);
    const double i = block_sum<kRedThreads>(im, sh);
    if (threadIdx.x == 0) {
        out[0] = r;
        out[1] = i;
    }
}

// lambda_y = sum_groups sum_terms coef * i^{#Y} s(y ^ f) psi_{y ^ f}
struct ObsDevTerm {
    uint64_t xmask, zmask;
    double coef;
    int32_t nY, pad;
};

template <typename C>
__global__ void __launch_bounds__(kRedThreads) k_apply_obs(const C* __restrict__ psi, C* __restrict__ lam, uint64_t N,
                                                           const ObsDevTerm* __restrict__ terms, int nterms) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t y = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; y < N; y += stride) {
        double re = 0.0, im = 0.0;
        for (int t = 0; t < nterms; t++) {
            const ObsDevTerm T = terms[t];
            const uint64_t y2 = y ^ T.xmask;
            double2 p = widen(psi[y2]);
            p = mul_ipow(p, T.nY + 2 * parity64(y2 & T.zmask));
            re = fma(T.coef, p.x, re);
            im = fma(T.coef, p.y, im);
        }
        lam[y] = narrow<C>(re, im);
    }
}

// double-float states: the same sum in double-float arithmetic on the FP32 pipes (exact
// products with the split coefficient, compensated sums)
struct ObsDevTermDF {
    uint64_t xmask, zmask;
    float ch, cl;  // coefficient = ch + cl
    int32_t nY, pad;
};

__global__ void __launch_bounds__(kRedThreads) k_apply_obs_df(const float4* __restrict__ psi, float4* __restrict__ lam,
                                                              uint64_t N, const ObsDevTermDF* __restrict__ terms,
                                                              int nterms) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t y = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; y < N; y += stride) {
        DFArith::Acc a = DFArith::zero();
        for (int t = 0; t < nterms; t++) {
            const ObsDevTermDF T = terms[t];
            const uint64_t y2 = y ^ T.xmask;
            const float4 v = DFArith::ipow(psi[y2], T.nY + 2 * parity64(y2 & T.zmask));
            DFArith::dprod(a.rs, a.rc, T.ch, T.cl, v.x, v.y);
            DFArith::dprod(a.is, a.ic, T.ch, T.cl, v.z, v.w);
        }
        lam[y] = DFArith::out(a);
    }
}

// ---------------------------------------------------------------- host side
// calls f(C*) with the state's buffer typed by its arithmetic layout
template <typename F>
void with_type(Arith ar, const void* p, F&& f) {
    switch (ar) {
        case Arith::F32: f(reinterpret_cast<const float2*>(p)); break;
        case Arith::F64: f(reinterpret_cast<const double2*>(p)); break;
        case Arith::DF: f(reinterpret_cast<const float4*>(p)); break;
    }
}
void ensure_scratch(qs_state* s, size_t part_doubles) {
    Scratch& sc = s->scratch;
    if (sc.part_cap < part_doubles) {
        if (sc.d_part) {
            if (s->pooled) {
                dev_free_async(sc.d_part, s->stream);
            } else {
                QS_TRY_CUDA(cudaStreamSynchronize(s->stream));
                dev_free(sc.d_part);
            }
            sc.d_part = nullptr;
            sc.part_cap = 0;
        }
        QS_TRY_CUDA(s->pooled ? dev_malloc_async(&sc.d_part, part_doubles * sizeof(double), s->stream)
                              : dev_malloc(&sc.d_part, part_doubles * sizeof(double)));
        sc.part_cap = part_doubles;
    }
    if (!sc.h_out && !s->pooled) {  // (a state of one call copies to pageable memory: no pinned allocation)
        QS_TRY_CUDA(host_malloc_pinned(&sc.h_out, 16 * sizeof(double)));
        sc.out_cap = 16;
    }
}

// final reduce of nslots partials into d_part[out_off..], copy 2 doubles to host, sync
void finish2(qs_state* s, int nslots, double out[2]) {
    // (straight into the pinned landing area, which the device can address, where there is one)
    double* d_out = s->pooled ? s->scratch.d_part + s->scratch.part_cap - 2 : s->scratch.h_out;
    k_final2<<<1, kRedThreads, 0, s->stream>>>(s->scratch.d_part, nslots, d_out);
    QS_TRY_CUDA(cudaGetLastError());
    if (s->pooled) {
        QS_TRY_CUDA(cudaMemcpyAsync(out, d_out, 2 * sizeof(double), cudaMemcpyDeviceToHost, s->stream));
        QS_TRY_CUDA(cudaStreamSynchronize(s->stream));
        return;
    }
    QS_TRY_CUDA(cudaStreamSynchronize(s->stream));
    out[0] = s->scratch.h_out[0];
    out[1] = s->scratch.h_out[1];
}

}  // namespace

std::vector<PauliGroup> group_observable(const qs_pauli_obs* obs, int n) {
    QS_REQUIRE(obs != nullptr, "null observable");
    QS_REQUIRE(obs->n_terms >= 0, "negative term count");
    QS_REQUIRE(obs->n_terms == 0 || (obs->coef && obs->x_mask && obs->z_mask), "null observable arrays");
    const uint64_t lim = n >= 64 ? ~0ull : ((1ull << n) - 1);
    std::map<uint64_t, size_t> idx;
    std::vector<PauliGroup> groups;
    for (int t = 0; t < obs->n_terms; t++) {
        QS_REQUIRE((obs->x_mask[t] & ~lim) == 0 && (obs->z_mask[t] & ~lim) == 0, "Pauli term acts on a qubit >= n");
        auto it = idx.find(obs->x_mask[t]);
        if (it == idx.end()) {
            idx[obs->x_mask[t]] = groups.size();
            groups.push_back(PauliGroup{obs->x_mask[t], {}, {}});
            it = idx.find(obs->x_mask[t]);
        }
        groups[it->second].coef.push_back(obs->coef[t]);
        groups[it->second].zmask.push_back(obs->z_mask[t]);
    }
    return groups;
}

void reduce_norm2(qs_state* s, double* out) {
    const uint64_t N = 1ull << s->n;
    const unsigned g = red_grid(N);
    ensure_scratch(s, 2 * g + 2);
    with_type(arith_of(s), s->data, [&](auto p) { k_norm2<<<g, kRedThreads, 0, s->stream>>>(p, N, s->scratch.d_part); });
    QS_TRY_CUDA(cudaGetLastError());
    double r[2];
    finish2(s, int(g), r);
    *out = r[0];
}

void reduce_inner(const qs_state* a, const qs_state* b, double out[2]) {
    qs_state* s = const_cast<qs_state*>(a);
    const uint64_t N = 1ull << s->n;
    const unsigned g = red_grid(N);
    ensure_scratch(s, 2 * g + 2);
    if (b->stream != s->stream) {
        // order b's pending work before the read on a's stream
        QS_TRY_CUDA(cudaStreamSynchronize(b->stream));
    }
    QS_REQUIRE(arith_of(a) == arith_of(b), "states in different layouts");
    with_type(arith_of(a), a->data, [&](auto pa) {
        using CP = decltype(pa);
        k_inner<<<g, kRedThreads, 0, s->stream>>>(pa, reinterpret_cast<CP>(b->data), N, s->scratch.d_part);
    });
    QS_TRY_CUDA(cudaGetLastError());
    finish2(s, int(g), out);
}

// Launches of one expectation: the tile passes, one launch per heavy chunk, and the terms that are
// alone in their flip group together (k_expect_singles): those that fit no tile, and one that a tile
// pass would stage the state for alone (whole calls, tile pass / single term: 173 / 142 us at n = 25 and
// 1138 / 801 us at n = 28 in complex128, 111 / 99 and 654 / 463 us in complex64; two terms take the tile
// pass, 740 us at n = 28 in complex64). With a
// cap on the block partials the grids shrink proportionally (the kernels loop over their work).
struct ExpectLaunches {
    std::vector<unsigned> pass_grid, heavy_grid;  // a diagonal observable: its one streaming pass in pass_grid
    std::vector<size_t> passes, heavy;            // indices into the plan
    std::vector<SingleTerm> singles;
    unsigned single_grid = 0;                     // blocks per single term
    size_t slots = 0;
};
SingleTerm single_term(const HeavyChunk& c) {
    SingleTerm t;
    t.f = c.g->xmask;
    t.z = c.g->zmask[c.t0];
    t.pivot = 63 - __builtin_clzll(t.f);
    const int nY = __builtin_popcountll(t.f & t.z);
    t.imag = nY & 1;
    t.coef = (((nY + 1) / 2) & 1) ? -2.0 * c.g->coef[c.t0] : 2.0 * c.g->coef[c.t0];
    return t;
}
ExpectLaunches expectation_launches(const ExpectPlan& plan, int n, Arith ar, size_t cap) {
    auto is_single = [&](const HeavyChunk& c) { return c.g->xmask && c.g->coef.size() == 1 && ar != Arith::DF; };
    ExpectLaunches L;
    if (plan.diag) L.pass_grid.push_back(expect_diag_grid(n, ar));
    for (size_t p = 0; p < plan.passes.size(); p++) {
        const auto& ch = plan.chunks[p];
        if (ch.size() == 1 && is_single(ch[0])) {
            L.singles.push_back(single_term(ch[0]));
            continue;
        }
        L.passes.push_back(p);
        L.pass_grid.push_back(expect_pass_grid(plan.passes[p], ar));
    }
    for (size_t h = 0; h < plan.heavy.size(); h++) {
        if (is_single(plan.heavy[h])) {
            L.singles.push_back(single_term(plan.heavy[h]));
            continue;
        }
        L.heavy.push_back(h);
        L.heavy_grid.push_back(red_grid((1ull << n) >> (plan.heavy[h].g->xmask ? 1 : 0)));
    }
    const size_t launches = L.pass_grid.size() + L.heavy_grid.size() + L.singles.size();
    if (!L.singles.empty()) {
        // eight pairs per thread, at most 256 blocks per term unless few terms leave the GPU idle (2432
        // blocks per term measured no faster on states beyond L2)
        const uint64_t want = ((1ull << (n - 1)) + kRedThreads * 8 - 1) / (kRedThreads * 8);
        const uint64_t most = std::max<uint64_t>(256, uint64_t(sms()) * 8 / L.singles.size());
        L.single_grid = unsigned(std::max<uint64_t>(1, std::min(want, most)));
    }
    size_t tot = L.singles.size() * size_t(L.single_grid);
    for (unsigned g : L.pass_grid) tot += g;
    for (unsigned g : L.heavy_grid) tot += g;
    if (tot > cap) {
        QS_REQUIRE(launches <= cap, "observable needs more kernel launches than the partial-sum scratch holds");
        const size_t per = cap / launches;
        for (unsigned& g : L.pass_grid) g = unsigned(std::min<size_t>(g, per));
        for (unsigned& g : L.heavy_grid) g = unsigned(std::min<size_t>(g, per));
        L.single_grid = unsigned(std::min<size_t>(L.single_grid, per));
    }
    for (unsigned g : L.pass_grid) L.slots += g;
    for (unsigned g : L.heavy_grid) L.slots += g;
    L.slots += L.singles.size() * size_t(L.single_grid);
    return L;
}

void launch_expectation(const ExpectPlan& plan, const ExpectLaunches& L, const void* psi, int n, Arith ar,
                        cudaStream_t st, double* part) {
    size_t slots = 0;
    if (plan.diag) {
        launch_expect_diag(plan.dp, psi, ar, part, L.pass_grid[0], st);
        return;
    }
    for (size_t p = 0; p < L.passes.size(); p++) {
        launch_expect_pass(plan.passes[L.passes[p]], psi, ar, part + 2 * slots, L.pass_grid[p], st);
        slots += L.pass_grid[p];
    }
    for (size_t t0 = 0; t0 < L.singles.size(); t0 += kMaxSingles) {
        SingleParams P;
        P.pairs = 1ull << (n - 1);
        const unsigned nt = unsigned(std::min<size_t>(kMaxSingles, L.singles.size() - t0));
        for (unsigned t = 0; t < nt; t++) P.t[t] = L.singles[t0 + t];
        const dim3 grid(L.single_grid, nt);
        if (ar == Arith::F32)
            k_expect_singles<float2, SingleAccF><<<grid, kRedThreads, 0, st>>>(static_cast<const float2*>(psi), P, part + 2 * slots);
        else
            k_expect_singles<double2, SingleAccD><<<grid, kRedThreads, 0, st>>>(static_cast<const double2*>(psi), P, part + 2 * slots);
        QS_TRY_CUDA(cudaGetLastError());
        slots += size_t(nt) * L.single_grid;
    }
    for (size_t h = 0; h < L.heavy.size(); h++) {
        const HeavyChunk& c = plan.heavy[L.heavy[h]];
        TermParams P;
        P.xmask = c.g->xmask;
        std::vector<int> fixed;
        if (P.xmask) fixed.push_back(__builtin_ctzll(P.xmask));
        P.ip = make_index_plan(n, fixed, 0);
        P.nterms = int(c.t1 - c.t0);
        for (size_t t = c.t0; t < c.t1; t++) {
            P.coef[t - c.t0] = c.g->coef[t];
            P.zmask[t - c.t0] = c.g->zmask[t];
            P.nY[t - c.t0] = __builtin_popcountll(c.g->xmask & c.g->zmask[t]);
        }
        with_type(ar, psi, [&](auto p) { k_expect_group<<<L.heavy_grid[h], kRedThreads, 0, st>>>(p, P, part + 2 * slots); });
        QS_TRY_CUDA(cudaGetLastError());
        slots += L.heavy_grid[h];
    }
}

void reduce_expectation(qs_state* s, const qs_pauli_obs* obs, double out[2]) {
    const std::vector<PauliGroup> groups = group_observable(obs, s->n);
    if (groups.empty()) {
        out[0] = out[1] = 0.0;
        return;
    }
    const ExpectPlan plan = plan_expectation(groups, s->n);
    const ExpectLaunches L = expectation_launches(plan, s->n, arith_of(s), size_t(1) << 40);
    ensure_scratch(s, 2 * L.slots + 2);
    launch_expectation(plan, L, s->data, s->n, arith_of(s), s->stream, s->scratch.d_part);
    finish2(s, int(L.slots), out);
}

void reduce_pauli_transition(qs_state* lam, const qs_state* psi, uint64_t xmask, uint64_t zmask, double out[2]) {
    const uint64_t N = 1ull << lam->n;
    const unsigned g = red_grid(N);
    ensure_scratch(lam, 2 * g + 2);
    const int nY = __builtin_popcountll(xmask & zmask);
    QS_REQUIRE(arith_of(lam) == arith_of(psi), "states in different layouts");
    with_type(arith_of(lam), lam->data, [&](auto pl) {
        using CP = decltype(pl);
        k_transition<<<g, kRedThreads, 0, lam->stream>>>(pl, reinterpret_cast<CP>(psi->data), N, xmask, zmask, nY,
                                                         lam->scratch.d_part);
    });
    QS_TRY_CUDA(cudaGetLastError());
    finish2(lam, int(g), out);
}

namespace {
// <bra|O|ket> of the X strings `xsum` and the groups `rest`
void transition_sum(const qs_state* bra, const std::vector<XsumParams>& xsum, const std::vector<PauliGroup>& rest,
                    const qs_state* ket, double out[2]) {
    qs_state* s = const_cast<qs_state*>(bra);
    const uint64_t N = 1ull << s->n;
    const Arith ar = arith_of(s);
    const ExpectPlan plan = rest.empty() ? ExpectPlan() : plan_transition(rest, s->n);
    std::vector<unsigned> grids, xgrids;
    size_t slots_needed = 0;
    for (const XsumParams& P : xsum) {
        xgrids.push_back(xsum_grid(P, ar));
        slots_needed += xgrids.back();
    }
    for (const TileParams& P : plan.passes) {
        grids.push_back(trans_pass_grid(P, ar));
        slots_needed += grids.back();
    }
    const unsigned gr = red_grid(N);
    slots_needed += size_t(gr) * plan.heavy.size();
    ensure_scratch(s, 2 * slots_needed + 2);
    size_t slots = 0;
    for (size_t p = 0; p < xsum.size(); p++) {
        launch_xsum(xsum[p], bra->data, ket->data, ar, s->scratch.d_part + 2 * slots, xgrids[p], s->stream);
        slots += xgrids[p];
    }
    for (size_t p = 0; p < plan.passes.size(); p++) {
        launch_transition_pass(plan.passes[p], bra->data, ket->data, ar, s->scratch.d_part + 2 * slots, grids[p],
                               s->stream);
        slots += grids[p];
    }
    // flip groups wider than a tile: one pass each
    for (const HeavyChunk& c : plan.heavy) {
        TermParams P;
        P.xmask = c.g->xmask;
        P.ip = make_index_plan(s->n, {}, 0);
        P.nterms = int(c.t1 - c.t0);
        for (size_t t = c.t0; t < c.t1; t++) {
            P.coef[t - c.t0] = c.g->coef[t];
            P.zmask[t - c.t0] = c.g->zmask[t];
            P.nY[t - c.t0] = __builtin_popcountll(c.g->xmask & c.g->zmask[t]);
        }
        double* part = s->scratch.d_part + 2 * slots;
        with_type(ar, s->data, [&](auto pb) {
            using CP = decltype(pb);
            k_transition_group<<<gr, kRedThreads, 0, s->stream>>>(pb, reinterpret_cast<CP>(ket->data), N, P, part);
        });
        QS_TRY_CUDA(cudaGetLastError());
        slots += gr;
    }
    finish2(s, int(slots), out);
}
}  // namespace

void reduce_transition(const qs_state* bra, const qs_pauli_obs* obs, const qs_state* ket, double out[2]) {
    const qs_state* s = bra;
    const std::vector<PauliGroup> groups = group_observable(obs, s->n);
    QS_REQUIRE(arith_of(bra) == arith_of(ket), "states in different layouts");
    if (ket->stream != s->stream) QS_TRY_CUDA(cudaStreamSynchronize(ket->stream));
    if (groups.empty()) {
        out[0] = out[1] = 0.0;
        return;
    }
    std::vector<XsumParams> xsum;
    const std::vector<PauliGroup> rest = split_xsum(groups, s->n, arith_of(s), xsum);
    transition_sum(bra, xsum, rest, ket, out);
    // ket components summed before their product with bra can leave FP32's range (from 2^124 on) where
    // the products do not: a result that is not finite is the tiled reads' to give
    if (!xsum.empty() && !(std::isfinite(out[0]) && std::isfinite(out[1]))) transition_sum(bra, {}, groups, ket, out);
}

void reduce_marginal(const qs_state* st, const int32_t* measured, double* out) {
    qs_state* s = const_cast<qs_state*>(st);
    FreeBits F;
    F.set = 0;
    F.nfree = F.nfix = 0;
    for (int q = 0; q < s->n; q++) {
        QS_REQUIRE(measured[q] >= 0 && measured[q] <= 2, "measured values must be 0, 1 or 2 (any)");
        F.nfree += measured[q] == 2;
        F.nfix += measured[q] != 2;
        if (measured[q] == 1) F.set |= 1ull << q;
    }
    F.insert = F.nfix < F.nfree ? 1 : 0;
    for (int q = 0, j = 0; q < s->n; q++)
        if ((measured[q] == 2) != (F.insert == 1)) F.pos[j++] = int8_t(q);
    const uint64_t work = 1ull << F.nfree;
    const unsigned g = red_grid(work);
    ensure_scratch(s, 2 * g + 2);
    with_type(arith_of(s), s->data, [&](auto p) { k_norm2_sub<<<g, kRedThreads, 0, s->stream>>>(p, F, s->scratch.d_part); });
    QS_TRY_CUDA(cudaGetLastError());
    double r[2];
    finish2(s, int(g), r);
    *out = r[0];
}

// Sampling: chunk masses (FP64), their cumulative sums in order on the host (a sequential sum, so
// that its rounding is one order whatever the GPU), then per sample the chunk by bisection and the
// index inside it. The mass pass also forms the segment sums that k_sample_pick reads where they
// save more than they cost: 370 us per 65536 chunks, against k_sample_find's 0.054 us per sample and
// about 60 us of its serial chain, so from count + 1024 >= chunks / 8 on. Whole calls, chunk search /
// segment sums: 194 / 157 us for 256 samples at n = 24, 126 / 65 us for 16 at n = 20; at n = 28,
// 1428 us for 4095 samples by the chunk search and 1578 us for 4096 with segment sums.

void sample_state(const qs_state* st, int count, const double* uniforms, uint64_t* out) {
    qs_state* s = const_cast<qs_state*>(st);
    if (count == 0) return;
    for (int k = 0; k < count; k++) QS_REQUIRE(uniforms[k] >= 0.0 && uniforms[k] < 1.0, "uniforms must lie in [0, 1)");
    const uint64_t N = 1ull << s->n;
    const int chunk_log = std::min(s->n, kSampleChunkLog);
    const uint64_t B = N >> chunk_log;
    bool segs = chunk_log == kSampleChunkLog && uint64_t(count) + 1024 >= B / 8;
    // one allocation: masses, cumulative masses, uniforms, residuals, chunks, results, segment sums
    // (1/64 of a complex128 state; without them where that much memory is not left)
    const size_t nc = size_t(count);
    const size_t doubles = B + (B + 1) + 4 * nc;
    double* d = nullptr;
    auto cleanup = [&]() {
        if (d) dev_free_async(d, s->stream);
    };
    try {
        if (segs && dev_malloc_async(reinterpret_cast<void**>(&d), (doubles + B * kSegsPerChunk) * sizeof(double),
                                     s->stream) != cudaSuccess) {
            cudaGetLastError();
            d = nullptr;
            segs = false;
        }
        if (!d) QS_TRY_CUDA(dev_malloc_async(reinterpret_cast<void**>(&d), doubles * sizeof(double), s->stream));
        double* d_mass = d;
        double* d_cum = d_mass + B;
        double* d_u = d_cum + (B + 1);
        double* d_resid = d_u + nc;
        uint64_t* d_chunk = reinterpret_cast<uint64_t*>(d_resid + nc);
        uint64_t* d_out = d_chunk + nc;
        float2* d_segs = reinterpret_cast<float2*>(d_out + nc);
        with_type(arith_of(s), s->data, [&](auto p) {
            using C = std::remove_const_t<std::remove_pointer_t<decltype(p)>>;
            if (segs)
                k_chunk_mass<C, true><<<unsigned(B), kRedThreads, 0, s->stream>>>(p, N, chunk_log, d_mass, d_segs);
            else
                k_chunk_mass<C, false><<<unsigned(B), kRedThreads, 0, s->stream>>>(p, N, chunk_log, d_mass, nullptr);
        });
        QS_TRY_CUDA(cudaGetLastError());
        QS_TRY_CUDA(cudaMemcpyAsync(d_u, uniforms, nc * sizeof(double), cudaMemcpyHostToDevice, s->stream));
        // cumulative distribution over chunks, in order, on the host
        std::vector<double> mass(B), cum(B + 1, 0.0);
        QS_TRY_CUDA(cudaMemcpyAsync(mass.data(), d_mass, B * sizeof(double), cudaMemcpyDeviceToHost, s->stream));
        QS_TRY_CUDA(cudaStreamSynchronize(s->stream));
        for (uint64_t b = 0; b < B; b++) cum[b + 1] = cum[b] + mass[b];
        const double total = cum[B];
        if (!(total > 0.0)) throw Error{QS_ERR_NUMERIC, "sampling a zero state"};
        uint64_t last = B - 1;
        while (last > 0 && !(mass[last] > 0.0)) last--;
        QS_TRY_CUDA(cudaMemcpyAsync(d_cum, cum.data(), (B + 1) * sizeof(double), cudaMemcpyHostToDevice, s->stream));
        k_sample_chunk<<<unsigned((nc + kRedThreads - 1) / kRedThreads), kRedThreads, 0, s->stream>>>(
            d_cum, B, d_u, total, last, count, d_chunk, d_resid);
        const unsigned blocks = unsigned((uint64_t(count) * 32 + kRedThreads - 1) / kRedThreads);
        with_type(arith_of(s), s->data, [&](auto p) {
            if (segs)
                k_sample_pick<<<blocks, kRedThreads, 0, s->stream>>>(p, N, d_chunk, d_resid, d_segs, count, d_out);
            else
                k_sample_find<<<blocks, kRedThreads, 0, s->stream>>>(p, N, chunk_log, d_chunk, d_resid, count, d_out);
        });
        QS_TRY_CUDA(cudaGetLastError());
        QS_TRY_CUDA(cudaMemcpyAsync(out, d_out, nc * sizeof(uint64_t), cudaMemcpyDeviceToHost, s->stream));
        QS_TRY_CUDA(cudaStreamSynchronize(s->stream));
    } catch (...) {
        cudaStreamSynchronize(s->stream);  // copies in flight may still read this call's host vectors
        cleanup();
        throw;
    }
    cleanup();
}

void launch_apply_observable(const std::vector<PauliGroup>& groups, const void* psi, void* lam, int n, Arith ar,
                             cudaStream_t st) {
    std::vector<ObsDevTerm> terms;
    for (const auto& g : groups)
        for (size_t t = 0; t < g.coef.size(); t++)
            terms.push_back(ObsDevTerm{g.xmask, g.zmask[t], g.coef[t], __builtin_popcountll(g.xmask & g.zmask[t]), 0});
    const uint64_t N = 1ull << n;
    if (terms.empty()) {
        QS_TRY_CUDA(cudaMemsetAsync(lam, 0, N * (ar == Arith::F32 ? 8 : 16), st));
        return;
    }
    ObsDevTerm* d_terms = nullptr;
    QS_TRY_CUDA(dev_malloc_async(reinterpret_cast<void**>(&d_terms), terms.size() * sizeof(ObsDevTerm), st));
    QS_TRY_CUDA(cudaMemcpyAsync(d_terms, terms.data(), terms.size() * sizeof(ObsDevTerm), cudaMemcpyHostToDevice, st));
    const unsigned g = red_grid(N);
    if (ar == Arith::DF) {
        std::vector<ObsDevTermDF> tdf(terms.size());
        for (size_t t = 0; t < terms.size(); t++) {
            tdf[t].xmask = terms[t].xmask;
            tdf[t].zmask = terms[t].zmask;
            split_double(terms[t].coef, tdf[t].ch, tdf[t].cl);
            tdf[t].nY = terms[t].nY;
            tdf[t].pad = 0;
        }
        static_assert(sizeof(ObsDevTermDF) <= sizeof(ObsDevTerm), "the term buffer holds either form");
        QS_TRY_CUDA(cudaMemcpyAsync(d_terms, tdf.data(), tdf.size() * sizeof(ObsDevTermDF), cudaMemcpyHostToDevice, st));
        QS_TRY_CUDA(cudaStreamSynchronize(st));  // tdf is host memory that dies on return
        k_apply_obs_df<<<g, kRedThreads, 0, st>>>(static_cast<const float4*>(psi), static_cast<float4*>(lam), N,
                                                  reinterpret_cast<const ObsDevTermDF*>(d_terms), int(terms.size()));
    } else {
        with_type(ar, psi, [&](auto pp) {
            using C = std::remove_const_t<std::remove_pointer_t<decltype(pp)>>;
            k_apply_obs<<<g, kRedThreads, 0, st>>>(pp, reinterpret_cast<C*>(lam), N, d_terms, int(terms.size()));
        });
    }
    QS_TRY_CUDA(cudaGetLastError());
    QS_TRY_CUDA(dev_free_async(d_terms, st));
}

}  // namespace qs

// ---------------------------------------------------------------- allocation-free variant
// Scratch for qs_expectation_noalloc: the per-block partial sums live in this fixed array
// instead of memory the library allocates. Every GPU that loads the library holds it (512 KiB)
// until the process exits. Host code may not use the symbol as a pointer; the device address
// is looked up once per device with cudaGetSymbolAddress.
namespace qs {

constexpr size_t kNoAllocScratchDoubles = size_t(1) << 16;
static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

namespace {
constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
double* g_noalloc_ptr[kMaxDevices] = {};

// device address of the scratch array on the current device (set up on first use there)
double* noalloc_scratch() {
    int dev = 0;
    QS_TRY_CUDA(cudaGetDevice(&dev));
    QS_REQUIRE(dev >= 0 && dev < kMaxDevices, "device index out of range");
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void* p = nullptr;
        QS_TRY_CUDA(cudaGetSymbolAddress(&p, g_noalloc_scratch));
        g_noalloc_ptr[dev] = static_cast<double*>(p);
    }
    return g_noalloc_ptr[dev];
}
}  // namespace

size_t noalloc_scratch_doubles() { return kNoAllocScratchDoubles; }

void expectation_noalloc(const void* psi, int n, qs_dtype dt, cudaStream_t st, const qs_pauli_obs* obs,
                         double out[2]) {
    QS_REQUIRE(psi != nullptr, "null state pointer");
    QS_REQUIRE((reinterpret_cast<uintptr_t>(psi) & 15) == 0, "state pointer must be 16-byte aligned");
    QS_REQUIRE(n >= 1 && n <= QS_MAX_QUBITS, "qubit count out of range (1..34)");
    QS_REQUIRE(dt == QS_C64 || dt == QS_C128, "unknown dtype");
    QS_REQUIRE(obs != nullptr && out != nullptr, "null observable or output");
    QS_REQUIRE(obs->n_terms >= 0, "negative term count");
    QS_REQUIRE(obs->n_terms == 0 || (obs->coef && obs->x_mask && obs->z_mask), "null observable arrays");
    const std::vector<PauliGroup> groups = group_observable(obs, n);
    if (groups.empty()) {
        out[0] = out[1] = 0.0;
        return;
    }
    const Arith ar = dt == QS_C64 ? Arith::F32 : Arith::F64;
    const ExpectPlan plan = plan_expectation(groups, n);
    // 2 doubles per block partial, plus the 2 final values at the end of the array
    const ExpectLaunches L = expectation_launches(plan, n, ar, (kNoAllocScratchDoubles - 2) / 2);
    double* scratch = noalloc_scratch();
    double* d_out = scratch + kNoAllocScratchDoubles - 2;
    launch_expectation(plan, L, psi, n, ar, st, scratch);
    const int slots = int(L.slots);
    k_final2<<<1, kRedThreads, 0, st>>>(scratch, slots, d_out);
    QS_TRY_CUDA(cudaGetLastError());
    QS_TRY_CUDA(cudaMemcpyAsync(out, d_out, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    QS_TRY_CUDA(cudaStreamSynchronize(st));
}

}  // namespace qs
