// Fused reverse steps of the adjoint gradient: for single-qubit rotations (below) and for runs of
// diagonal gates (second half of the file). A rotation is
// R_P(theta) = exp(+i theta P / 2), P in {X, Y} (the paper's gate table sign).
//
// At gate j of the reverse sweep psi holds psi_j (the state after the gate) and lambda holds
// lambda_j = U_{j+1}^+ ... U_G^+ H psi_G. Then dE/dtheta_j = -Im <lambda_j|P|psi_j>; afterwards
// both buffers are multiplied by R_P(theta)^+. Both are done pair by pair: each contributes
// conj(lambda) * (P psi) to the block's partial sum, then the 2x2 adjoint is applied to the pair in
// psi and in lambda; several rotations share a pass over the state. Per-block partials land in their own
// slots (deterministic); one final kernel reduces every gate's slots.
#include <algorithm>

#include "qsim_arith.cuh"

namespace qs {

namespace {

constexpr int kAdjThreads = 256;

// accumulators of Im conj(l) * p for each arithmetic policy, FP64-class in all three
template <typename P>
struct GradAcc;

template <>
struct GradAcc<NativeArith<double>> {
    double im = 0.0;
    __device__ void add(double2 l, double2 p) {
        im = fma(l.x, p.y, im);
        im = fma(-l.y, p.x, im);
    }
    __device__ double imag() const { return im; }
};

template <>
struct GradAcc<NativeArith<float>> {
    DFAcc im;
    __device__ GradAcc() { df_zero(im); }
    __device__ void add(float2 l, float2 p) {
        df_add_prod(im, l.x, p.y);
        df_add_prod(im, -l.y, p.x);
    }
    __device__ double imag() const { return df_value(im); }
};

// the imaginary part of an FP32-pair gradient accumulator as its unevaluated pair (s, c)
__device__ __forceinline__ void acc_pair(const GradAcc<NativeArith<float>>& g, float& s, float& c) {
    s = g.im.hi;
    c = g.im.lo;
}

template <typename P>
__device__ __forceinline__ void rot_step(typename P::C& a, typename P::C& b, typename P::C& la, typename P::C& lb,
                                         int axis, const typename P::K* U, GradAcc<P>& g) {
    if (axis == 1) {
        g.add(la, b);
        g.add(lb, a);
    } else {
        g.add(la, P::ipow(b, 3));
        g.add(lb, P::ipow(a, 1));
    }
    typename P::Acc r0 = P::first(U[0], a), r1 = P::first(U[2], a), s0 = P::first(U[0], la), s1 = P::first(U[2], la);
    P::mac(r0, U[1], b);
    P::mac(r1, U[3], b);
    P::mac(s0, U[1], lb);
    P::mac(s1, U[3], lb);
    a = P::out(r0);
    b = P::out(r1);
    la = P::out(s0);
    lb = P::out(s1);
}

// One thread's partial of a rotation as 8 bytes, and sums of such: FP32 pairs, or an FP64 value for
// the FP64 policy. (On GB300 FP64 warp stages, or a conversion in every lane, cost microseconds per
// launch: FP32 pairs stay pairs until one FP64 conversion per block.)
template <typename P>
struct GradSlot {
    using T = float2;
    __device__ __forceinline__ static T zero() { return make_float2(0.f, 0.f); }
    __device__ __forceinline__ static T of(const GradAcc<P>& g) {
        T t;
        acc_pair(g, t.x, t.y);
        return t;
    }
    __device__ __forceinline__ static T add(T a, T b) {
        float h, e;
        DFArith::two_sum(a.x, b.x, h, e);
        return make_float2(h, __fadd_rn(a.y, __fadd_rn(b.y, e)));
    }
    __device__ __forceinline__ static T down(T a, int o) {
        return make_float2(__shfl_down_sync(0xffffffffu, a.x, o), __shfl_down_sync(0xffffffffu, a.y, o));
    }
    __device__ __forceinline__ static double value(T a) { return double(a.x) + double(a.y); }
};
template <>
struct GradSlot<NativeArith<double>> {
    using T = double;
    __device__ __forceinline__ static T zero() { return 0.0; }
    __device__ __forceinline__ static T of(const GradAcc<NativeArith<double>>& g) { return g.imag(); }
    __device__ __forceinline__ static T add(T a, T b) { return a + b; }
    __device__ __forceinline__ static T down(T a, int o) { return __shfl_down_sync(0xffffffffu, a, o); }
    __device__ __forceinline__ static double value(T a) { return a; }
};

// One rotation's reverse step on a pair of a tile: the gradient partial, then R^+ on both buffers.
template <typename P>
struct TileRot {
    using C = typename P::C;
    using Acc = GradAcc<P>;
    __device__ __forceinline__ static C order(const C& v) { return v; }  // global <-> tile element
    __device__ __forceinline__ static void step(C& a, C& b, C& la, C& lb, int axis, const typename P::K* U, Acc& g) {
        rot_step<P>(a, b, la, lb, axis, U, g);
    }
    __device__ __forceinline__ static typename GradSlot<P>::T slot(const Acc& g) { return GradSlot<P>::of(g); }
};
// Double-float: tile elements {re_hi, im_hi, re_lo, im_lo}, real and imaginary parts as packed pairs. The
// entries of R^+ are real multiples of 1 and i (X: [[c, -i s], [-i s, c]]; Y: [[c, -s], [s, c]]), so every
// component is a sum of two real products.
template <>
struct TileRot<DFArith> {
    using C = float4;
    struct Acc {
        float2 s = make_float2(0.f, 0.f), c = make_float2(0.f, 0.f);
    };
    __device__ __forceinline__ static C order(const C& v) { return make_float4(v.x, v.z, v.y, v.w); }
    __device__ __forceinline__ static Pair2 pair(const C& v) { return Pair2{make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
    __device__ __forceinline__ static Pair2 neg(const Pair2& v) {
        return Pair2{make_float2(-v.h.x, -v.h.y), make_float2(-v.l.x, -v.l.y)};
    }
    __device__ __forceinline__ static Pair2 conj_swap(const Pair2& v) {  // (im, -re)
        return Pair2{make_float2(v.h.y, -v.h.x), make_float2(v.l.y, -v.l.x)};
    }
    // (pair_dot gives {re_hi, re_lo, im_hi, im_lo})
    __device__ __forceinline__ static C dot(float2 xh, float2 xl, const Pair2& a, float2 yh, float2 yl, const Pair2& b) {
        return order(pair_dot(xh, xl, a, yh, yl, b));
    }
    __device__ __forceinline__ static void update(C& a, C& b, int axis, float ch, float cl, float sh, float sl) {
        const Pair2 va = pair(a), vb = pair(b);
        const float2 c2 = make_float2(ch, ch), c2l = make_float2(cl, cl);
        if (axis == 1) {  // a' = c a - i s b, b' = -i s a + c b
            const float2 s2 = make_float2(sh, -sh), s2l = make_float2(sl, -sl);
            a = dot(c2, c2l, va, s2, s2l, swapped(vb));
            b = dot(s2, s2l, swapped(va), c2, c2l, vb);
        } else {  // a' = c a - s b, b' = s a + c b
            const float2 s2 = make_float2(sh, sh), s2l = make_float2(sl, sl);
            const float2 m2 = make_float2(-sh, -sh), m2l = make_float2(-sl, -sl);
            a = dot(c2, c2l, va, m2, m2l, vb);
            b = dot(s2, s2l, va, c2, c2l, vb);
        }
    }
    __device__ __forceinline__ static void grad(Acc& g, const Pair2& l, const Pair2& p) {
        dprod2(g.s, g.c, l.h, l.l, p.h, p.l, false);
    }
    __device__ __forceinline__ static void step(C& a, C& b, C& la, C& lb, int axis, const float4* U, Acc& g) {
        const Pair2 va = pair(a), vb = pair(b), wa = pair(la), wb = pair(lb);
        if (axis == 1) {  // Im conj(la) b + Im conj(lb) a
            grad(g, wa, conj_swap(vb));
            grad(g, wb, conj_swap(va));
        } else {  // Y psi = (-i b, i a): Re conj(lb) a - Re conj(la) b
            grad(g, wb, va);
            grad(g, neg(wa), vb);
        }
        // c = Re U[0]; s = -Im U[1] (X) or -Re U[1] (Y)
        const float ch = U[0].x, cl = U[0].y;
        const float sh = axis == 1 ? -U[1].z : -U[1].x, sl = axis == 1 ? -U[1].w : -U[1].y;
        update(a, b, axis, ch, cl, sh, sl);
        update(la, lb, axis, ch, cl, sh, sl);
    }
    __device__ __forceinline__ static float2 slot(const Acc& g) {
        float h, e;
        DFArith::two_sum(g.s.x, g.s.y, h, e);
        return make_float2(h, __fadd_rn(e, __fadd_rn(g.c.x, g.c.y)));
    }
};

// Consecutive reverse steps for rotations on distinct qubits q_0 (the latest in the circuit), q_1, ...
// in one pass: a tile of psi and of lambda (2^t amplitudes each, t <= kAdjTileBits local qubits that
// hold every q_r) stays in shared memory while, two rotations at a time, each thread takes the gradient
// partials of a group of four amplitudes and un-applies both rotations in registers. (The rotations
// commute, so each gradient is the same whichever others are already un-applied.) Partials of rotation r
// go to part[r grid .. (r + 1) grid).
// What bounds it: double-float arithmetic (about 110 FP32 operations per amplitude and rotation, on packed
// pairs) and, per pass, about 20 us of reads, writes and a second wave that is two thirds full (1024
// tiles on 608 CTA slots at n = 20). A layer of 20 RY rotations at n = 20: ten passes of two rotations
// 150 us, three passes here 137 us with scalar double-float updates and 124 us with packed pairs (46 us
// for eight rotations). Four CTAs per SM (64 registers, 150 bytes spilled) and three (85) differ by less
// than the runs.
constexpr int kAdjTileBits = 10;
template <typename P>
struct AdjTileParams {
    uint64_t n_tiles;
    uint64_t dep_hi[1 << (kAdjTileBits - 8)];  // address bits of local bits 8..t-1
    int32_t t, nr;
    uint8_t lq[kAdjTileBits];                  // local bit -> qubit, ascending
    uint8_t bit[kAdjMaxRotations];             // local bit of rotation r
    uint8_t axis[kAdjMaxRotations];
    typename P::K U[kAdjMaxRotations][4];      // R_r^+
};

template <typename P>
__global__ void __launch_bounds__(kAdjThreads, 4) k_adj_tile(typename P::C* __restrict__ psi, typename P::C* __restrict__ lam,
                                                             const __grid_constant__ AdjTileParams<P> A, double* part) {
    using C = typename P::C;
    using R = TileRot<P>;
    using S = GradSlot<P>;
    using T = typename S::T;
    extern __shared__ __align__(16) unsigned char adj_smem[];
    const uint32_t tid = threadIdx.x, N = 1u << A.t;
    C* sp = reinterpret_cast<C*>(adj_smem);
    C* sl = sp + N;
    T* acc = reinterpret_cast<T*>(sl + N);  // [rotation][thread]
    for (int r = 0; r < A.nr; r++) acc[r * kAdjThreads + tid] = S::zero();
    uint64_t off = 0;
#pragma unroll 1
    for (int b = 0; b < A.t && b < 8; b++)
        if ((tid >> b) & 1u) off |= 1ull << A.lq[b];
    for (uint64_t tile = blockIdx.x; tile < A.n_tiles; tile += gridDim.x) {
        uint64_t base = tile;
#pragma unroll 1
        for (int b = 0; b < A.t; b++) {
            const uint64_t lo = base & ((1ull << A.lq[b]) - 1ull);
            base = ((base ^ lo) << 1) | lo;
        }
        C* gp = psi + (base | off);
        C* gl = lam + (base | off);
        constexpr int kU = (1 << kAdjTileBits) / kAdjThreads;
        {
            C v[kU], u[kU];
#pragma unroll
            for (int k = 0; k < kU; k++)
                if (tid + k * kAdjThreads < N) {
                    v[k] = gp[A.dep_hi[k]];
                    u[k] = gl[A.dep_hi[k]];
                }
#pragma unroll
            for (int k = 0; k < kU; k++)
                if (tid + k * kAdjThreads < N) {
                    sp[tid + k * kAdjThreads] = R::order(v[k]);
                    sl[tid + k * kAdjThreads] = R::order(u[k]);
                }
        }
        __syncthreads();
        for (int r = 0; r < A.nr; r += 2) {
            if (r + 1 < A.nr) {
                const int b0 = A.bit[r], b1 = A.bit[r + 1];
                const int blo = min(b0, b1), bhi = max(b0, b1);
                if (tid < N / 4) {  // N / 4 <= kAdjThreads
                    const uint32_t l = insert_zero(insert_zero(tid, blo), bhi);
                    const uint32_t m0 = 1u << b0, m1 = 1u << b1;
                    C v[4] = {sp[l], sp[l | m0], sp[l | m1], sp[l | m0 | m1]};
                    C u[4] = {sl[l], sl[l | m0], sl[l | m1], sl[l | m0 | m1]};
                    typename R::Acc g0, g1;
                    R::step(v[0], v[1], u[0], u[1], A.axis[r], A.U[r], g0);
                    R::step(v[2], v[3], u[2], u[3], A.axis[r], A.U[r], g0);
                    R::step(v[0], v[2], u[0], u[2], A.axis[r + 1], A.U[r + 1], g1);
                    R::step(v[1], v[3], u[1], u[3], A.axis[r + 1], A.U[r + 1], g1);
                    sp[l] = v[0];
                    sp[l | m0] = v[1];
                    sp[l | m1] = v[2];
                    sp[l | m0 | m1] = v[3];
                    sl[l] = u[0];
                    sl[l | m0] = u[1];
                    sl[l | m1] = u[2];
                    sl[l | m0 | m1] = u[3];
                    T* a = acc + r * kAdjThreads + tid;
                    a[0] = S::add(a[0], R::slot(g0));
                    a[kAdjThreads] = S::add(a[kAdjThreads], R::slot(g1));
                }
            } else {
                const uint32_t m0 = 1u << A.bit[r];
                typename R::Acc g;
                for (uint32_t j = tid; j < N / 2; j += kAdjThreads) {
                    const uint32_t l = insert_zero(j, A.bit[r]);
                    C a = sp[l], b = sp[l | m0], la = sl[l], lb = sl[l | m0];
                    R::step(a, b, la, lb, A.axis[r], A.U[r], g);
                    sp[l] = a;
                    sp[l | m0] = b;
                    sl[l] = la;
                    sl[l | m0] = lb;
                }
                T* a = acc + r * kAdjThreads + tid;
                a[0] = S::add(a[0], R::slot(g));
            }
            __syncthreads();
        }
#pragma unroll
        for (int k = 0; k < kU; k++)
            if (tid + k * kAdjThreads < N) {
                gp[A.dep_hi[k]] = R::order(sp[tid + k * kAdjThreads]);
                gl[A.dep_hi[k]] = R::order(sl[tid + k * kAdjThreads]);
            }
    }
    __syncthreads();
    // rotation r's sum over the block by warp r mod 8, in a fixed order
    const uint32_t lane = tid & 31u;
    for (int r = int(tid >> 5); r < A.nr; r += kAdjThreads / 32) {
        T v = acc[r * kAdjThreads + lane];
        for (int k = 1; k < kAdjThreads / 32; k++) v = S::add(v, acc[r * kAdjThreads + lane + 32 * k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = S::add(v, S::down(v, o));
        if (lane == 0) part[size_t(r) * gridDim.x + blockIdx.x] = S::value(v);
    }
}

// out[s] = sum of part[s * nb .. s * nb + nb) in a fixed order, one block per slot
__global__ void __launch_bounds__(kAdjThreads) k_slot_sums(const double* __restrict__ part, int nb, double* out) {
    __shared__ double sh[kAdjThreads / 32];
    double v = 0.0;
    for (int j = threadIdx.x; j < nb; j += kAdjThreads) v += part[size_t(blockIdx.x) * nb + j];
    const double r = block_sum<kAdjThreads>(v, sh);
    if (threadIdx.x == 0) out[blockIdx.x] = r;
}

// ---- reverse step for a run of diagonal gates
// Diagonal gates commute with each other and with every diagonal Pauli string P (a Z string),
// so for a parametric gate exp(i theta P / 2) inside a run of diagonal gates,
// <lambda_j|P|psi_j> = <lambda|P|psi> with psi, lambda taken after the whole run: one pass
// computes every such gradient of the run and then multiplies both buffers by the run's inverse
// (the product of the conjugated diagonals). Each factor of that product is either a table over
// up to 6 qubits (applied where a condition on other bits holds) or a sign (-1)^popc(x & zmask).
// FP64-class running sums: double for the FP64 policy, an FP32 (sum, compensation) pair
// (Knuth TwoSum) for the FP32 and double-float policies
template <typename P>
struct RedSum {
    float s = 0.f, c = 0.f;
    __device__ void add(float ws, float wc, bool neg) {
        if (neg) { ws = -ws; wc = -wc; }
        float h, e;
        DFArith::two_sum(s, ws, h, e);
        s = h;
        c = __fadd_rn(c, __fadd_rn(e, wc));
    }
    __device__ void add(const RedSum& o, bool neg) { add(o.s, o.c, neg); }
    __device__ double value() const { return double(s) + double(c); }
};
template <>
struct RedSum<NativeArith<double>> {
    double v = 0.0;
    __device__ void add(const RedSum& o, bool neg) { v += neg ? -o.v : o.v; }
    __device__ double value() const { return v; }
};
// Im(conj(l) p) of one amplitude as a RedSum
__device__ __forceinline__ RedSum<DFArith> im_conj_prod(float4 l, float4 p, RedSum<DFArith>) {
    RedSum<DFArith> w;
    DFArith::dprod0(w.s, w.c, l.x, l.y, p.z, p.w);
    DFArith::dprod(w.s, w.c, -l.z, -l.w, p.x, p.y);
    return w;
}
__device__ __forceinline__ RedSum<NativeArith<float>> im_conj_prod(float2 l, float2 p, RedSum<NativeArith<float>>) {
    RedSum<NativeArith<float>> w;
    DFArith::dprod0(w.s, w.c, l.x, 0.f, p.y, 0.f);
    DFArith::dprod(w.s, w.c, -l.y, 0.f, p.x, 0.f);
    return w;
}
__device__ __forceinline__ RedSum<NativeArith<double>> im_conj_prod(double2 l, double2 p, RedSum<NativeArith<double>>) {
    RedSum<NativeArith<double>> w;
    w.v = fma(l.x, p.y, -l.y * p.x);
    return w;
}

// The Walsh-Hadamard transform of one value per lane: lane l ends with the sum over lanes s of
// (-1)^{popc(s & l)} v_s (five butterfly stages across the warp, (a + b, a - b) per lane pair).
template <typename P>
__device__ __forceinline__ RedSum<P> lane_wht(RedSum<P> v, int lane) {
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        RedSum<P> o;
        o.s = __shfl_xor_sync(0xffffffffu, v.s, m);
        o.c = __shfl_xor_sync(0xffffffffu, v.c, m);
        const bool hi = (lane & m) != 0;  // this lane takes o - v, its partner v + o
        RedSum<P> r = hi ? o : v;
        r.add(hi ? v : o, hi);
        v = r;
    }
    return v;
}
template <>
__device__ __forceinline__ RedSum<NativeArith<double>> lane_wht(RedSum<NativeArith<double>> v, int lane) {
#pragma unroll
    for (int m = 1; m < 32; m <<= 1) {
        const double o = __shfl_xor_sync(0xffffffffu, v.v, m);
        v.v = (lane & m) ? o - v.v : v.v + o;
    }
    return v;
}
template <typename P>
__device__ __forceinline__ RedSum<P> lane_fetch(const RedSum<P>& v, int src) {
    RedSum<P> o;
    o.s = __shfl_sync(0xffffffffu, v.s, src);
    o.c = __shfl_sync(0xffffffffu, v.c, src);
    return o;
}
template <>
__device__ __forceinline__ RedSum<NativeArith<double>> lane_fetch(const RedSum<NativeArith<double>>& v, int src) {
    RedSum<NativeArith<double>> o;
    o.v = __shfl_sync(0xffffffffu, v.v, src);
    return o;
}

__device__ __forceinline__ float4 kmul(float4 a, float4 b) { return DFArith::out(DFArith::first(a, b)); }
__device__ __forceinline__ float2 kmul(float2 a, float2 b) { return cmul(a, b); }
__device__ __forceinline__ double2 kmul(double2 a, double2 b) { return cmul(a, b); }
template <typename K>
__device__ __forceinline__ K kone();
template <>
__device__ __forceinline__ float4 kone<float4>() { return make_float4(1.f, 0.f, 0.f, 0.f); }
template <>
__device__ __forceinline__ float2 kone<float2>() { return make_float2(1.f, 0.f); }
template <>
__device__ __forceinline__ double2 kone<double2>() { return make_double2(1.0, 0.0); }

// f and sign times factor F at x
template <typename K>
__device__ __forceinline__ void adj_diag_factor(const AdjDiagFactor& F, uint64_t x, const K* stab, K& f, int& sign) {
    if ((x & F.cond_mask) != F.cond_val) return;
    sign ^= parity64(x & F.zmask);
    if (F.pair_shift) sign ^= parity64(x & (x >> F.pair_shift) & F.pair_mask);
    if (F.sign_only) {
        sign ^= 1;
    } else if (F.tab_off >= 0) {
        uint32_t li = 0;
        for (int b = 0; b < F.nrun; b++) {
            const uint32_t c = F.run[b];
            li |= (uint32_t(x >> (c & 0xFFu)) & ((1u << ((c >> 8) & 0xFFu)) - 1u)) << (c >> 16);
        }
        f = kmul(f, stab[F.tab_off + int(li)]);
    }
}

constexpr int kDiagKA = 4;  // amplitudes per thread between two gradient flushes

// Thread t of T = grid x 256 threads takes the amplitudes x = j T + t, kDiagKA values of j at a
// time, each giving w_x = Im(conj(lam_x) psi_x). Per j the warp transforms its 32 values
// (Walsh-Hadamard across the lanes), and lane g takes the coefficient at its gradient term's Z
// bits among the lane bits, with the sign of the rest of the term's Z bits: every term of the
// run from one transform, so the per-amplitude cost does not grow with the number of gradients.
// Factors on the bits of t alone (below log2 T) are multiplied once per thread, not per amplitude.
// What bounds it: instruction issue. A layer's RZ gates and CZ ladder, every factor per amplitude / the
// low ones per thread: complex128 38.4 / 28.2 us at n = 20 (926 / 635 instructions per amplitude) and
// 135 / 86 us at n = 22, complex64 27.5 / 20.4 us at n = 20.
template <typename P>
__global__ void __launch_bounds__(kAdjThreads) k_adj_diag(typename P::C* __restrict__ psi, typename P::C* __restrict__ lam,
                                                           const typename P::K* __restrict__ tab,
                                                           const __grid_constant__ AdjDiagParams A, double* part) {
    using C = typename P::C;
    using K = typename P::K;
    using R = RedSum<P>;
    extern __shared__ __align__(16) unsigned char adj_smem[];
    K* stab = reinterpret_cast<K*>(adj_smem);
    R* wred = reinterpret_cast<R*>(adj_smem + ((size_t(A.ntab) * sizeof(K) + 15) & ~size_t(15)));  // [warp][g]
    for (int i = threadIdx.x; i < A.ntab; i += kAdjThreads) stab[i] = tab[i];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t T = uint64_t(gridDim.x) * kAdjThreads;
    const uint64_t t = uint64_t(blockIdx.x) * kAdjThreads + threadIdx.x;
    const uint64_t J = (A.n_amp + T - 1) / T;
    const uint64_t gz = lane < A.ng ? A.gz[lane] : 0;
    R gsum;  // lane g: this warp's sum for gradient term g
    const uint64_t t0 = t - uint64_t(lane);  // the warp's first thread
    K f_low = kone<K>();
    int sign_low = 0;
#pragma unroll 1
    for (int k = 0; k < A.nlow; k++) adj_diag_factor(A.f[k], t, stab, f_low, sign_low);
    for (uint64_t j0 = 0; j0 < J; j0 += kDiagKA) {
        R acc[kDiagKA];
#pragma unroll
        for (int j = 0; j < kDiagKA; j++) {
            const uint64_t x = (j0 + j) * T + t;
            if (j0 + j >= J || x >= A.n_amp) continue;
            C p = psi[x], l = lam[x];
            if (A.ng) acc[j] = im_conj_prod(l, p, R());
            K f = f_low;
            int sign = sign_low;
#pragma unroll 1
            for (int k = A.nlow; k < A.nf; k++) adj_diag_factor(A.f[k], x, stab, f, sign);
            p = P::out(P::first(f, p));
            l = P::out(P::first(f, l));
            if (sign) {
                p = P::ipow(p, 2);
                l = P::ipow(l, 2);
            }
            psi[x] = p;
            lam[x] = l;
        }
        if (A.ng) {
            // gradient term g over the warp's 32 amplitudes of item j, x = (j0 + j) T + t0 + s:
            // the lane bits s, the warp's bits of t0 and the item's bits of (j0 + j) T are
            // disjoint (T is a power of two), so the sign (-1)^{popc(x & z_g)} factors into
            // (-1)^{popc(s & z_g)}, whose sum over s is the warp's Walsh-Hadamard coefficient at
            // z_g mod 32, times the sign of the rest
#pragma unroll
            for (int j = 0; j < kDiagKA; j++) {
                const R w = lane_fetch(lane_wht(acc[j], lane), int(gz & 31u));
                if (lane < A.ng && j0 + j < J) gsum.add(w, parity64(((j0 + j) * T + t0) & gz) != 0);
            }
        }
    }
    if (A.ng) {
        if (lane < A.ng) wred[warp * 32 + lane] = gsum;
        __syncthreads();
        if (threadIdx.x < A.ng) {
            R total;
            for (int w = 0; w < kAdjThreads / 32; w++) total.add(wred[w * 32 + threadIdx.x], false);
            part[size_t(threadIdx.x) * gridDim.x + blockIdx.x] = total.value();
        }
    }
}

size_t adj_diag_smem(int ntab, Arith ar) {
    const size_t rs = ar == Arith::F64 ? sizeof(double) : 2 * sizeof(float);
    return ((size_t(ntab) * kernel_entry_bytes(ar) + 15) & ~size_t(15)) + rs * (kAdjThreads / 32) * 32;
}

// R_P(theta)^+ = cos(theta/2) I - i sin(theta/2) P as a row-major 2x2 matrix, P = X (axis 1) or Y
void rot_dagger(int axis, double theta, cplx (&U)[4]) {
    const double c = std::cos(theta / 2), s = std::sin(theta / 2);
    if (axis == 1) { U[0] = c; U[1] = cplx(0, -s); U[2] = cplx(0, -s); U[3] = c; }
    else { U[0] = c; U[1] = -s; U[2] = s; U[3] = c; }
}

// qubits 0 and 1 always lie in the tile: runs of 64 bytes (double-float)
uint64_t adj_low(int n) { return (1ull << std::min(n, 2)) - 1; }

template <typename P>
void launch_tile(void* psi, void* lam, int n, int nr, const int* qubit, const int* axis, const double* theta, double* part,
                 unsigned grid, cudaStream_t st) {
    AdjTileParams<P> A;
    const int t = std::min(n, kAdjTileBits);
    uint64_t local = adj_low(n);
    for (int r = 0; r < nr; r++) local |= 1ull << qubit[r];
    for (int q = 0; q < n && __builtin_popcountll(local) < t; q++) local |= 1ull << q;
    QS_REQUIRE(__builtin_popcountll(local) == t, "rotations of a pass on too many qubits");
    int loc_of[64], k = 0;
    for (int q = 0; q < n; q++)
        if ((local >> q) & 1) {
            loc_of[q] = k;
            A.lq[k++] = uint8_t(q);
        }
    A.t = t;
    A.nr = nr;
    A.n_tiles = 1ull << (n - t);
    for (int h = 0; h < (1 << (kAdjTileBits - 8)); h++) {
        A.dep_hi[h] = 0;
        for (int b = 8; b < t; b++)
            if ((h >> (b - 8)) & 1) A.dep_hi[h] |= 1ull << A.lq[b];
    }
    for (int r = 0; r < nr; r++) {
        A.bit[r] = uint8_t(loc_of[qubit[r]]);
        A.axis[r] = uint8_t(axis[r]);
        cplx U[4];
        rot_dagger(axis[r], theta[r], U);
        for (int e = 0; e < 4; e++) A.U[r][e] = P::host_k(U[e].real(), U[e].imag());
    }
    const size_t smem = 2 * (sizeof(typename P::C) << t) + sizeof(typename GradSlot<P>::T) * kAdjThreads * size_t(nr);
    static PerDevice setup;
    setup.once([](int) {
        constexpr size_t most = 2 * (sizeof(typename P::C) << kAdjTileBits) + 8 * kAdjThreads * kAdjMaxRotations;
        QS_TRY_CUDA(cudaFuncSetAttribute(k_adj_tile<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(most)));
    });
    k_adj_tile<P><<<grid, kAdjThreads, smem, st>>>(reinterpret_cast<typename P::C*>(psi),
                                                   reinterpret_cast<typename P::C*>(lam), A, part);
}

}  // namespace

unsigned adj_grid(int n) {
    const uint64_t pairs = 1ull << (n - 1);
    // a power of two (the diagonal-run kernel's amplitude partition relies on it)
    uint64_t want = 1;
    while (want * 2 * kAdjThreads <= pairs && want < 1024) want *= 2;
    return unsigned(want);
}

bool adjoint_rotations_fit(uint64_t qubits, int n) {
    return __builtin_popcountll(qubits) <= kAdjMaxRotations &&
           __builtin_popcountll(qubits | adj_low(n)) <= std::min(n, kAdjTileBits);
}

void launch_adjoint_rotations(void* psi, void* lam, int n, Arith ar, int nr, const int* qubit, const int* axis,
                              const double* theta, double* part, unsigned grid, cudaStream_t st) {
    QS_REQUIRE(nr >= 1 && nr <= kAdjMaxRotations, "rotations per pass out of range");
    for (int r = 0; r < nr; r++) QS_REQUIRE(axis[r] == 1 || axis[r] == 2, "rotations that share a pass are about X or Y");
    switch (ar) {
        case Arith::F32: launch_tile<NativeArith<float>>(psi, lam, n, nr, qubit, axis, theta, part, grid, st); break;
        case Arith::F64: launch_tile<NativeArith<double>>(psi, lam, n, nr, qubit, axis, theta, part, grid, st); break;
        case Arith::DF: launch_tile<DFArith>(psi, lam, n, nr, qubit, axis, theta, part, grid, st); break;
    }
    QS_TRY_CUDA(cudaGetLastError());
}

void launch_adjoint_diag(void* psi, void* lam, int n, Arith ar, const void* tab, const AdjDiagParams& run, double* part,
                         unsigned grid, cudaStream_t st) {
    AdjDiagParams A = run;
    const uint64_t T = uint64_t(grid) * kAdjThreads;
    auto low = [&](const AdjDiagFactor& f) {
        uint64_t bits = f.cond_mask | f.zmask | f.pair_mask | (f.pair_mask << f.pair_shift);
        for (int j = 0; j < f.nq; j++) bits |= 1ull << f.q[j];
        return bits < T;
    };
    // (signs commute exactly; in complex64 the tables keep their order, another one would change the
    // product's last bit)
    AdjDiagFactor* const end = A.f + A.nf;
    if (ar == Arith::F32)
        std::stable_partition(A.f, end, [](const AdjDiagFactor& f) { return f.tab_off >= 0; });
    else
        std::stable_partition(A.f, end, low);
    A.nlow = int(std::find_if_not(A.f, end, low) - A.f);
    const size_t smem = adj_diag_smem(A.ntab, ar);
    switch (ar) {
        case Arith::F32:
            k_adj_diag<NativeArith<float>><<<grid, kAdjThreads, smem, st>>>(
                static_cast<float2*>(psi), static_cast<float2*>(lam), static_cast<const float2*>(tab), A, part);
            break;
        case Arith::F64:
            k_adj_diag<NativeArith<double>><<<grid, kAdjThreads, smem, st>>>(
                static_cast<double2*>(psi), static_cast<double2*>(lam), static_cast<const double2*>(tab), A, part);
            break;
        case Arith::DF:
            k_adj_diag<DFArith><<<grid, kAdjThreads, smem, st>>>(
                static_cast<float4*>(psi), static_cast<float4*>(lam), static_cast<const float4*>(tab), A, part);
            break;
    }
    QS_TRY_CUDA(cudaGetLastError());
}

void launch_slot_sums(const double* part, int nslots, unsigned nb, double* out, cudaStream_t st) {
    if (nslots <= 0) return;
    k_slot_sums<<<nslots, kAdjThreads, 0, st>>>(part, int(nb), out);
    QS_TRY_CUDA(cudaGetLastError());
}

}  // namespace qs
