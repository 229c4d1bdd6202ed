// Several gates in one pass over the state (gate-by-gate runs): each gate keeps its own update
// (Eq. update_mat; diagonal, Pauli and swap forms), applied one after the other to a tile of the
// state held in shared memory.
//
// A pass has a set L of at most t "local" qubits. A tile is the 2^t amplitudes whose other qubits
// are fixed; a CTA stages it, applies the pass's gates in order and writes it back, so the pass
// costs one read and one write of the state whatever its gate count. Only the qubits a gate changes
// (dense targets, X or Y positions, swapped qubits) must lie in L: controls, phases, diagonals and Z
// factors on other qubits are fixed bits of the tile's base.
//
// What bounds it: small states by host work and launches (one per pass instead of one per gate), large
// complex128 states by double-float arithmetic (86 FP32 operations per amplitude and general one-qubit
// gate), large complex64 states by shared-memory traffic and index work, each instead of HBM.
// Measured, random U3 + CZ circuits of depth 10 gate by gate, one pass per gate / several: complex128
// 783 / 142 us at n = 12 (175 gates), 1047 / 197 us at n = 16, 5.11 / 4.36 ms at n = 22, 1936 / 1434 ms
// at n = 30; complex64 1168 / 302 us at n = 18, 50.4 / 20.5 ms at n = 26, 913 / 368 ms at n = 30.
// Two CTAs per SM (106 registers) measured 2 % faster than three and 3 % faster than four (spills);
// staging the gate records in shared memory instead of the parameter bank gave 31 -> 29 us per pass at
// n = 12 and lost 7 % in complex64 at n = 26, so the records stay in the parameter bank.
//
// Passes are formed on the host by list scheduling: the gates in order, each taken when it commutes
// with every gate skipped before it (no shared qubit, or only diagonal action on the shared ones)
// and its changed qubits fit L. In complex64 a pass ends at the first gate that does not fit: every
// amplitude then sees its gates in circuit order with the roundings of single launches (an FP32 value
// computed from the state would otherwise change in its seventh digit with the order).
#include <algorithm>
#include <memory>

#include "qsim_arith.cuh"

namespace qs {

namespace {

constexpr int kPassThreads = 256;
constexpr int kPassMaxBits = 12;

// pair kinds (one barrier each), then elementwise kinds (runs of them share one sweep)
enum PassKind : uint8_t { kPassD1, kPassD2, kPassFlip, kPassRot, kPassSwap, kPassSign, kPassPhase, kPassDiag, kPassZSign, kPassZRot };
constexpr uint8_t kPassFirstElementwise = kPassSign;

// one gate in the tile's coordinates: l is a tile-local index, base the tile's fixed bits
struct PassOp {
    uint8_t kind = 0;
    uint8_t m = 0;            // kPassDiag: index bits
    uint8_t mode = 0;         // kPassD1: 0 general, 1 real, 2 real diagonal and imaginary off-diagonal;
                              // kPassPhase: i^mode, 0 general; kPassFlip, kPassRot: number of Y
    uint8_t t0 = 0, t1 = 0;   // local positions (targets; pivot of a flip)
    uint8_t run = 1;          // elementwise: gates in the sweep that starts here
    uint16_t data = 0;        // first entry in the pool
    uint32_t lcm = 0, lcv = 0;  // acts where (l & lcm) == lcv ...
    uint32_t lx = 0, lz = 0;  // local flip and Z masks
    uint64_t ncm = 0, ncv = 0;  // ... and (base & ncm) == ncv
    uint64_t nz = 0;          // Z mask on the tile's fixed bits
    uint8_t pos[QS_MAX_TARGETS] = {};  // kPassDiag: local position of index bit j, or 128 + qubit
    uint8_t pad[2] = {};
};

template <typename P, int NOP, int NDATA>
struct PassParams {
    uint64_t n_tiles;
    uint64_t dep_hi[1 << (kPassMaxBits - 8)];  // address bits of local bits 8..t-1
    int32_t t, nops;
    int32_t ieee_in, ieee_out;                 // double-float: the buffer holds / gets IEEE doubles
    uint8_t lq[kPassMaxBits];                  // local bit -> qubit, ascending
    PassOp op[NOP];
    typename P::K data[NDATA];
};

// (a, b) <- K (a, b). In FP64 and double-float, real matrices and those with a real diagonal and an imaginary
// off-diagonal (mode 1, 2) skip the products by zero.
template <typename P>
__device__ __forceinline__ void pass_pair(const typename P::K* K, int, typename P::C& a, typename P::C& b) {
    typename P::Acc r0 = P::first(K[0], a), r1 = P::first(K[2], a);
    P::mac(r0, K[1], b);
    P::mac(r1, K[3], b);
    a = P::out(r0);
    b = P::out(r1);
}
// The general complex update on packed pairs: 92 + 8 register swaps for a pair instead of 172 instructions.
__device__ __forceinline__ float4 df_mul_add2(const float4& k0, const float4& k1, const Pair2& a, const Pair2& as,
                                              const Pair2& b, const Pair2& bs) {
    float2 s, c;
    dprod2(s, c, make_float2(k0.x, k0.x), make_float2(k0.y, k0.y), a.h, a.l, true);
    dprod2(s, c, make_float2(-k0.z, k0.z), make_float2(-k0.w, k0.w), as.h, as.l, false);
    dprod2(s, c, make_float2(k1.x, k1.x), make_float2(k1.y, k1.y), b.h, b.l, false);
    dprod2(s, c, make_float2(-k1.z, k1.z), make_float2(-k1.w, k1.w), bs.h, bs.l, false);
    const float2 h = __fadd2_rn(s, c), bp = sub2(h, s);
    const float2 l = __fadd2_rn(sub2(s, sub2(h, bp)), sub2(c, bp));
    return make_float4(h.x, l.x, h.y, l.y);
}
template <>
__device__ __forceinline__ void pass_pair<DFArith>(const float4* K, int mode, float4& a, float4& b) {
    const Pair2 va{make_float2(a.x, a.z), make_float2(a.y, a.w)}, vb{make_float2(b.x, b.z), make_float2(b.y, b.w)};
    auto dup = [](float f) { return make_float2(f, f); };
    auto mp = [](float f) { return make_float2(-f, f); };
    if (mode == 0) {
        const Pair2 wa = swapped(va), wb = swapped(vb);
        a = df_mul_add2(K[0], K[1], va, wa, vb, wb);
        b = df_mul_add2(K[2], K[3], va, wa, vb, wb);
    } else if (mode == 1) {
        a = pair_dot(dup(K[0].x), dup(K[0].y), va, dup(K[1].x), dup(K[1].y), vb);
        b = pair_dot(dup(K[2].x), dup(K[2].y), va, dup(K[3].x), dup(K[3].y), vb);
    } else {  // i y b = (-y b.im, y b.re)
        const Pair2 wa = swapped(va), wb = swapped(vb);
        a = pair_dot(dup(K[0].x), dup(K[0].y), va, mp(K[1].z), mp(K[1].w), wb);
        b = pair_dot(mp(K[2].z), mp(K[2].w), wa, dup(K[3].x), dup(K[3].y), vb);
    }
}
template <>
__device__ __forceinline__ void pass_pair<NativeArith<double>>(const double2* K, int mode, double2& a, double2& b) {
    using P = NativeArith<double>;
    double2 ra, rb;
    if (mode == 0) {
        ra = P::first(K[0], a);
        rb = P::first(K[2], a);
        P::mac(ra, K[1], b);
        P::mac(rb, K[3], b);
    } else if (mode == 1) {
        ra = make_double2(fma(K[1].x, b.x, K[0].x * a.x), fma(K[1].x, b.y, K[0].x * a.y));
        rb = make_double2(fma(K[3].x, b.x, K[2].x * a.x), fma(K[3].x, b.y, K[2].x * a.y));
    } else {
        ra = make_double2(fma(-K[1].y, b.y, K[0].x * a.x), fma(K[1].y, b.x, K[0].x * a.y));
        rb = make_double2(fma(K[3].x, b.x, -K[2].y * a.y), fma(K[3].x, b.y, K[2].y * a.x));
    }
    a = ra;
    b = rb;
}

// a tile holds double-float amplitudes as {re_hi, im_hi, re_lo, im_lo}: the packed pairs of
// pass_pair are then aligned register pairs of one 16-byte access
__device__ __forceinline__ float4 tile_order(float4 v) { return make_float4(v.x, v.z, v.y, v.w); }
__device__ __forceinline__ float2 tile_order(float2 v) { return v; }
__device__ __forceinline__ double2 tile_order(double2 v) { return v; }
template <typename C>
struct Tile {
    C* s;
    __device__ __forceinline__ C get(uint32_t l) const { return tile_order(s[l]); }
    __device__ __forceinline__ void put(uint32_t l, C v) const { s[l] = tile_order(v); }
};

// k v, rounded as k_phase and k_diag do
template <typename P>
__device__ __forceinline__ typename P::C pass_mul(const typename P::K& k, const typename P::C& v) {
    typename P::Acc a = P::zero();
    P::mac(a, k, v);
    return P::out(a);
}
template <>
__device__ __forceinline__ float4 pass_mul<DFArith>(const float4& k, const float4& v) {
    return DFArith::out(DFArith::first(k, v));
}

template <typename P>
__device__ __forceinline__ void pass_elementwise(typename P::C& v, int& sign, const PassOp& o,
                                                 const typename P::K* data, uint32_t l, uint64_t base) {
    if ((base & o.ncm) != o.ncv) return;
    const bool on = (l & o.lcm) == o.lcv;
    if (o.kind == kPassSign) {
        sign ^= on ? 1 : 0;
        return;
    }
    if (!on) return;
    switch (o.kind) {
        case kPassPhase:
            v = o.mode == 0 ? pass_mul<P>(data[o.data], v) : P::ipow(v, o.mode);
            break;
        case kPassDiag: {
            uint32_t r = 0;
            for (int j = 0; j < o.m; j++) {
                const int p = o.pos[j];
                r |= uint32_t(p < 128 ? (l >> p) & 1u : uint32_t(base >> (p - 128)) & 1u) << j;
            }
            v = pass_mul<P>(data[o.data + r], v);
            break;
        }
        case kPassZSign:
            sign ^= (__popc(l & o.lz) + __popcll(base & o.nz)) & 1;
            break;
        default:  // kPassZRot
            v = P::out(P::first(data[o.data + ((__popc(l & o.lz) + __popcll(base & o.nz)) & 1)], v));
            break;
    }
}

template <typename P, int NOP, int NDATA>
__global__ void __launch_bounds__(kPassThreads, 2) k_gate_pass(typename P::C* __restrict__ psi,
                                                            const __grid_constant__ PassParams<P, NOP, NDATA> A) {
    using C = typename P::C;
    extern __shared__ __align__(16) unsigned char pass_smem[];
    const uint32_t tid = threadIdx.x, T = 1u << A.t;
    const Tile<C> s{reinterpret_cast<C*>(pass_smem)};
    uint64_t off = 0;  // address bits of this thread's local bits 0..7
#pragma unroll 1
    for (int b = 0; b < A.t && b < 8; b++)
        if ((tid >> b) & 1u) off |= 1ull << A.lq[b];
    constexpr int kU = 4;  // loads in flight per thread
    for (uint64_t tile = blockIdx.x; tile < A.n_tiles; tile += gridDim.x) {
        uint64_t base = tile;
#pragma unroll 1
        for (int b = 0; b < A.t; b++) {
            const uint64_t lo = base & ((1ull << A.lq[b]) - 1ull);
            base = ((base ^ lo) << 1) | lo;
        }
        C* p = psi + (base | off);
        for (uint32_t l0 = tid; l0 < T; l0 += kU * kPassThreads) {
            C v[kU];
#pragma unroll
            for (int u = 0; u < kU; u++)
                if (l0 + u * kPassThreads < T) v[u] = p[A.dep_hi[(l0 + u * kPassThreads) >> 8]];
#pragma unroll
            for (int u = 0; u < kU; u++) {
                if (l0 + u * kPassThreads >= T) break;
                if constexpr (std::is_same<P, DFArith>::value) {
                    if (A.ieee_in) {
                        const double2 d = *reinterpret_cast<const double2*>(&v[u]);
                        split_double_int(d.x, v[u].x, v[u].y);
                        split_double_int(d.y, v[u].z, v[u].w);
                    }
                }
                s.put(l0 + u * kPassThreads, v[u]);
            }
        }
        __syncthreads();
        for (int i = 0; i < A.nops;) {
            const PassOp& o = A.op[i];
            if (o.kind >= kPassFirstElementwise) {
                const int e = i + o.run;
                for (uint32_t l = tid; l < T; l += kPassThreads) {
                    C v = s.get(l);
                    int sign = 0;  // the sweep's factors -1 (CZ, Z strings), applied once
                    for (int k = i; k < e; k++) pass_elementwise<P>(v, sign, A.op[k], A.data, l, base);
                    if (sign) v = P::ipow(v, 2);
                    s.put(l, v);
                }
                i = e;
            } else {
                i++;
                if ((base & o.ncm) != o.ncv) continue;
                const typename P::K* k = A.data + o.data;
                switch (o.kind) {
                    case kPassD1: {
                        const uint32_t bit = 1u << o.t0;
                        for (uint32_t j = tid; j < T / 2; j += kPassThreads) {
                            const uint32_t l = insert_zero(j, o.t0);
                            if ((l & o.lcm) != o.lcv) continue;
                            C a = s.get(l), b = s.get(l | bit);
                            pass_pair<P>(k, o.mode, a, b);
                            s.put(l, a);
                            s.put(l | bit, b);
                        }
                        break;
                    }
                    case kPassD2: {
                        const int plo = min(o.t0, o.t1), phi = max(o.t0, o.t1);
                        const uint32_t b0 = 1u << o.t0, b1 = 1u << o.t1;
                        for (uint32_t j = tid; j < T / 4; j += kPassThreads) {
                            const uint32_t l = insert_zero(insert_zero(j, plo), phi);
                            if ((l & o.lcm) != o.lcv) continue;
                            const uint32_t x[4] = {l, l | b0, l | b1, l | b0 | b1};
                            C v[4];
#pragma unroll
                            for (int w = 0; w < 4; w++) v[w] = s.get(x[w]);
#pragma unroll 1
                            for (int z = 0; z < 4; z++) {
                                typename P::Acc a = P::first(k[4 * z], v[0]);
#pragma unroll
                                for (int w = 1; w < 4; w++) P::mac(a, k[4 * z + w], v[w]);
                                s.put(l | ((z & 1) ? b0 : 0u) | ((z & 2) ? b1 : 0u), P::out(a));
                            }
                        }
                        break;
                    }
                    case kPassSwap: {
                        const int plo = min(o.t0, o.t1), phi = max(o.t0, o.t1);
                        const uint32_t ba = 1u << o.t0, bb = 1u << o.t1;
                        for (uint32_t j = tid; j < T / 4; j += kPassThreads) {
                            const uint32_t l = insert_zero(insert_zero(j, plo), phi);
                            if ((l & o.lcm) != o.lcv) continue;
                            const C a = s.get(l | ba);
                            s.put(l | ba, s.get(l | bb));
                            s.put(l | bb, a);
                        }
                        break;
                    }
                    default: {  // kPassFlip, kPassRot: pairs (l, l ^ lx), the pivot bit t0 clear in l
                        const int pn = __popcll(base & o.nz);
                        for (uint32_t j = tid; j < T / 2; j += kPassThreads) {
                            const uint32_t l = insert_zero(j, o.t0), l2 = l ^ o.lx;
                            if ((l & o.lcm) != o.lcv) continue;
                            const int par = (__popc(l & o.lz) + pn) & 1, par2 = (__popc(l2 & o.lz) + pn) & 1;
                            const C a = s.get(l), b = s.get(l2);
                            if (o.kind == kPassFlip) {
                                s.put(l2, P::ipow(a, o.mode + 2 * par));
                                s.put(l, P::ipow(b, o.mode + 2 * par2));
                            } else {  // entries cos, +- i^(1 + nY) sin
                                const bool imag = !(o.mode & 1);
                                s.put(l, RotMix<P>::mix(k[0], k[1 + par2], imag, a, b));
                                s.put(l2, RotMix<P>::mix(k[0], k[1 + par], imag, b, a));
                            }
                        }
                        break;
                    }
                }
            }
            __syncthreads();
        }
        for (uint32_t l = tid; l < T; l += kPassThreads) {
            C v = s.get(l);
            if constexpr (std::is_same<P, DFArith>::value) {
                if (A.ieee_out) {
                    reinterpret_cast<double2*>(p)[A.dep_hi[l >> 8]] = make_double2(join_df_int(v.x, v.y), join_df_int(v.z, v.w));
                    continue;
                }
            }
            p[A.dep_hi[l >> 8]] = v;
        }
    }
}

// ------------------------------------------------------------------ host: scheduling
// the qubits an op changes and those it only reads (commuting with anything diagonal there)
struct OpQubits {
    uint64_t x = 0, d = 0;
};
OpQubits op_qubits(const Op& op) {
    OpQubits q;
    uint64_t t = 0;
    for (int v : op.targets) t |= 1ull << v;
    for (int v : op.controls) q.d |= 1ull << v;
    switch (op.kind) {
        case OpKind::Dense:
        case OpKind::Swap: q.x = t; break;
        case OpKind::Diag: q.d |= t; break;
        case OpKind::Phase: break;
        case OpKind::Pauli:
        case OpKind::PauliRot:
            q.x = op.xmask;
            q.d |= op.zmask & ~op.xmask;
            break;
    }
    return q;
}
bool is_identity(const Op& op) {
    return (op.kind == OpKind::Phase && op.phase == cplx(1.0, 0.0)) ||
           (op.kind == OpKind::Pauli && op.xmask == 0 && op.zmask == 0);
}
// What an op costs as a launch of its own and inside a tile pass, which adds kPassBase for the staging,
// in full passes of the lightest kind (an X gate's launch: 356 us at n = 26, 90 at n = 24, 21 at n = 22
// in complex128, 175 / 48 / 12 us in complex64). From runs of 1, 2, 3, 4 and 8 gates of a kind on low qubits,
// as launches and as one pass, at n = 20, 22, 24 and 26; the figures lean to the launches where the sizes
// differ. One launch each / one pass, microseconds for 8 gates at n = 26 (F64 at n = 24): double-float
// U3 2849 / 2239, RY 2855 / 1386, dense pair 3207 / 3794, RZ 2737 / 2862, rotation 2880 / 1716, CZ 1202 /
// 1035, X 2749 / 1184; complex64 U3 1336 / 516, dense pair 1501 / 873, RZ 1448 / 1467, CZ 765 / 589; F64
// U3 2098 / 1882, RZ 1051 / 1201, rotation 1432 / 1541. A tile pass gains nothing per diagonal factor (index
// and parity work per amplitude and gate) and, in double-float, nothing per dense pair (arithmetic).
enum OpClass { kOpD1, kOpD1Half, kOpD2, kOpSign, kOpFactor, kOpSwap, kOpFlip, kOpRot, kOpClasses };
struct ClassCost {
    double alone, inside;
};
constexpr ClassCost kClassCost[3][kOpClasses] = {  // by Arith
    {{1.0, kPassGateInside[0]}, {1.0, 0.45}, {1.3, 0.75}, {1.1, 0.38}, {1.05, 1.1}, {1.9, 0.35}, {1.05, 0.45}, {1.05, 0.5}},    // F32
    {{2.9, kPassGateInside[1]}, {1.5, 1.4}, {5.8, 5.0}, {1.0, 0.2}, {1.45, 1.5}, {1.6, 0.25}, {1.0, 0.3}, {2.0, 2.1}},         // F64
    {{1.0, kPassGateInside[2]}, {1.0, 0.45}, {1.15, 1.25}, {1.2, 0.28}, {1.0, 1.0}, {1.4, 0.25}, {0.95, 0.38}, {1.05, 0.55}},  // DF
};
static_assert(int(Arith::F32) == 0 && int(Arith::F64) == 1 && int(Arith::DF) == 2, "order of kClassCost");
constexpr double kPassBase[3] = {0.95, 1.1, 1.1};
OpClass op_class(const Op& op) {
    switch (op.kind) {
        case OpKind::Dense: {
            if (op.targets.size() > 1) return kOpD2;
            const auto& d = op.data;
            const bool re = d[0].imag() == 0.0 && d[3].imag() == 0.0;
            const bool half = re && ((d[1].imag() == 0.0 && d[2].imag() == 0.0) || (d[1].real() == 0.0 && d[2].real() == 0.0));
            return half ? kOpD1Half : kOpD1;
        }
        case OpKind::Swap: return kOpSwap;
        case OpKind::Diag: return kOpFactor;
        case OpKind::Phase: return op.phase.real() == 0.0 || op.phase.imag() == 0.0 ? kOpSign : kOpFactor;
        case OpKind::Pauli: return op.xmask ? kOpFlip : kOpSign;
        default: return op.xmask ? kOpRot : kOpFactor;
    }
}
ClassCost op_pass_cost(const Op& op, Arith ar) {
    ClassCost c = kClassCost[int(ar)][op_class(op)];
    // a launch touches the share of the state that its controls select; on the lowest qubits it still
    // moves most of the lines
    for (int q : op.controls) c.alone *= ar == Arith::F32 ? (q < 4 ? 0.9 : 0.55) : (q < 3 ? 0.8 : 0.5);
    if (op.kind == OpKind::Swap) c.alone *= 0.5;
    // a launch reads a long string's amplitudes further apart (X or Y on 13 qubits: 1.2 to 1.6)
    if (op.kind == OpKind::PauliRot && op.xmask) c.alone += 0.03 * (__builtin_popcountll(op.xmask) - 2);
    return c;
}
constexpr int kPassOps = 128, kPassData = 640;      // a pass's limits (16.5 KB of parameters)
constexpr int kPassOpsS = 24, kPassDataS = 96;      // the small form's (3.2 KB)
size_t pass_entries(const Op& op) {
    switch (op.kind) {
        case OpKind::Dense:
        case OpKind::Diag: return op.data.size();
        case OpKind::Phase: return 1;
        case OpKind::PauliRot: return 3;
        default: return 0;
    }
}

template <typename P, int NOP, int NDATA>
void launch_pass_t(const Op* const* ops, int nops, uint64_t local, void* psi, int n, bool ieee_in, bool ieee_out,
                   cudaStream_t st) {
    auto Ap = std::make_unique<PassParams<P, NOP, NDATA>>();
    PassParams<P, NOP, NDATA>& A = *Ap;
    int loc_of[64];
    int t = 0;
    for (int q = 0; q < n; q++) {
        loc_of[q] = -1;
        if (!((local >> q) & 1)) continue;
        loc_of[q] = t;
        A.lq[t++] = uint8_t(q);
    }
    A.t = t;
    A.n_tiles = 1ull << (n - t);
    A.ieee_in = ieee_in ? 1 : 0;
    A.ieee_out = ieee_out ? 1 : 0;
    for (int h = 0; h < (1 << (kPassMaxBits - 8)); h++) {
        A.dep_hi[h] = 0;
        for (int b = 8; b < t; b++)
            if ((h >> (b - 8)) & 1) A.dep_hi[h] |= 1ull << A.lq[b];
    }
    auto local_mask = [&](uint64_t m) {
        uint32_t r = 0;
        for (int b = 0; b < t; b++)
            if ((m >> A.lq[b]) & 1) r |= 1u << b;
        return r;
    };
    int nd = 0;
    auto put = [&](cplx v) { A.data[nd++] = P::host_k(v.real(), v.imag()); };
    for (int i = 0; i < nops; i++) {
        const Op& op = *ops[i];
        PassOp o;
        o.data = uint16_t(nd);
        uint64_t cm = 0, cv = 0;
        for (size_t j = 0; j < op.controls.size(); j++) {
            cm |= 1ull << op.controls[j];
            if (op.cvals[j]) cv |= 1ull << op.controls[j];
        }
        o.lcm = local_mask(cm);
        o.lcv = local_mask(cv);
        o.ncm = cm & ~local;
        o.ncv = cv & ~local;
        switch (op.kind) {
            case OpKind::Dense: {
                o.kind = op.targets.size() == 1 ? kPassD1 : kPassD2;
                o.t0 = uint8_t(loc_of[op.targets[0]]);
                if (op.targets.size() == 2) o.t1 = uint8_t(loc_of[op.targets[1]]);
                for (const cplx& v : op.data) put(v);
                if (o.kind == kPassD1) {
                    const auto& d = op.data;
                    const bool diag_re = d[0].imag() == 0.0 && d[3].imag() == 0.0;
                    if (diag_re && d[1].imag() == 0.0 && d[2].imag() == 0.0) o.mode = 1;
                    else if (diag_re && d[1].real() == 0.0 && d[2].real() == 0.0) o.mode = 2;
                }
                break;
            }
            case OpKind::Swap:
                o.kind = kPassSwap;
                o.t0 = uint8_t(loc_of[op.targets[0]]);
                o.t1 = uint8_t(loc_of[op.targets[1]]);
                break;
            case OpKind::Phase:
                o.kind = kPassPhase;
                if (op.phase == cplx(0.0, 1.0)) o.mode = 1;
                if (op.phase == cplx(-1.0, 0.0)) o.kind = kPassSign;
                if (op.phase == cplx(0.0, -1.0)) o.mode = 3;
                put(op.phase);
                break;
            case OpKind::Diag:
                o.kind = kPassDiag;
                o.m = uint8_t(op.targets.size());
                for (size_t j = 0; j < op.targets.size(); j++) {
                    const int q = op.targets[j];
                    o.pos[j] = uint8_t(loc_of[q] >= 0 ? loc_of[q] : 128 + q);
                }
                for (const cplx& v : op.data) put(v);
                break;
            case OpKind::Pauli:
            case OpKind::PauliRot: {
                const bool rot = op.kind == OpKind::PauliRot;
                o.lx = local_mask(op.xmask);
                o.lz = local_mask(op.zmask);
                o.nz = op.zmask & ~local;
                o.mode = uint8_t(__builtin_popcountll(op.xmask & op.zmask) & 3);
                const double c = std::cos(op.angle / 2), sn = std::sin(op.angle / 2);
                if (op.xmask) {
                    o.kind = rot ? kPassRot : kPassFlip;
                    o.t0 = uint8_t(__builtin_ctz(o.lx));
                    if (rot) {  // cos, i^(1 + nY) sin, its negative
                        const int e = (1 + o.mode) & 3;
                        const cplx k(e == 0 ? sn : e == 2 ? -sn : 0.0, e == 1 ? sn : e == 3 ? -sn : 0.0);
                        put(c);
                        put(k);
                        put(-k);
                    }
                } else {
                    o.kind = rot ? kPassZRot : kPassZSign;
                    if (rot) {
                        put(cplx(c, sn));
                        put(cplx(c, -sn));
                    }
                }
                break;
            }
        }
        A.op[i] = o;
    }
    A.nops = nops;
    for (int i = 0; i < nops;) {  // sweeps of consecutive elementwise gates
        if (A.op[i].kind < kPassFirstElementwise) {
            i++;
            continue;
        }
        int e = i;
        while (e < nops && A.op[e].kind >= kPassFirstElementwise) e++;
        A.op[i].run = uint8_t(e - i);
        i = e;
    }
    const size_t smem = sizeof(typename P::C) << t;
    const unsigned grid = unsigned(std::min<uint64_t>(A.n_tiles, uint64_t(device_sms()) * 8));
    k_gate_pass<P, NOP, NDATA><<<grid, kPassThreads, smem, st>>>(reinterpret_cast<typename P::C*>(psi), A);
    QS_TRY_CUDA(cudaGetLastError());
}

template <typename P>
void launch_pass_p(const Op* const* ops, int nops, size_t ndata, uint64_t local, void* psi, int n, bool in, bool out,
                   cudaStream_t st) {
    if (nops <= kPassOpsS && ndata <= size_t(kPassDataS))
        launch_pass_t<P, kPassOpsS, kPassDataS>(ops, nops, local, psi, n, in, out, st);
    else
        launch_pass_t<P, kPassOps, kPassData>(ops, nops, local, psi, n, in, out, st);
}

}  // namespace

// Tile bits: up to a 32 KB tile (fewer passes) once 2^8 tiles fill the SMs, never below 8 (9 in FP32)
// bits: under that the extra passes cost more than the wider spread over SMs gives. Whole calls of the
// depth-10 U3 + CZ circuit (and of four repetitions of RZ RX RZ + CNOT layers) with at least 7 / 8 / 9 / 10
// bits: complex128 142 / 137 / 147 / 199 us (186 / 174 / 203 / 288) at n = 12, 173 / 162 / 173 / 226 (220 / 212 /
// 236 / 335) at n = 14; complex64, whose passes end with the first gate that does not fit, 195 / 180 / 166 /
// 175 (216 / 203 / 212 / 270) at n = 12 and 230 / 220 / 199 / 203 (257 / 240 / 251 / 324) at n = 14.
int gate_pass_bits(int n, Arith ar) {
    const int most = ar == Arith::F32 ? 12 : 11, least = ar == Arith::F32 ? 9 : 8;
    return std::min(n, std::max(least, std::min(most, n - 8)));
}

std::vector<GatePass> schedule_passes(const std::vector<Op>& ops, int n, Arith ar) {
    const int t = gate_pass_bits(n, ar);
    // 64-byte runs per tile row
    const uint64_t low = (1ull << std::min(n, ar == Arith::F32 ? 3 : 2)) - 1;
    auto fits_alone = [&](const Op& op, const OpQubits& q) {
        if (op.kind == OpKind::Dense && op.targets.size() > 2) return false;
        return __builtin_popcountll(q.x | low) <= t;
    };
    std::vector<GatePass> out;
    constexpr size_t kWindow = 512;  // gates looked at together: bounds the host time of long runs
    std::vector<OpQubits> q(ops.size());
    for (size_t i = 0; i < ops.size(); i++) q[i] = op_qubits(ops[i]);
    std::vector<size_t> rem, keep;
    size_t next = 0;
    auto refill = [&]() {
        while (rem.size() < kWindow && next < ops.size()) {
            if (!is_identity(ops[next])) rem.push_back(next);
            next++;
        }
    };
    for (refill(); !rem.empty(); refill()) {
        GatePass p;
        if (!fits_alone(ops[rem[0]], q[rem[0]])) {
            p.ops.push_back(rem[0]);
            p.alone = op_pass_cost(ops[rem[0]], ar).alone;
            out.push_back(std::move(p));
            rem.erase(rem.begin());
            continue;
        }
        uint64_t L = low, bx = 0, bd = 0;
        size_t data = 0;
        keep.clear();
        bool ended = false;
        for (size_t i : rem) {
            const Op& op = ops[i];
            const size_t e = pass_entries(op);
            if (!ended && (q[i].x & (bx | bd)) == 0 && (q[i].d & bx) == 0 && p.ops.size() < size_t(kPassOps) &&
                data + e <= size_t(kPassData) && __builtin_popcountll(L | q[i].x) <= t && fits_alone(op, q[i])) {
                L |= q[i].x;
                data += e;
                const ClassCost cost = op_pass_cost(op, ar);
                p.alone += cost.alone;
                p.inside += cost.inside;
                p.ops.push_back(i);
            } else {
                bx |= q[i].x;
                bd |= q[i].d;
                keep.push_back(i);
                ended = ar == Arith::F32;
            }
        }
        for (int b = 0; b < n && __builtin_popcountll(L) < t; b++) L |= 1ull << b;
        p.local = L;
        p.data = data;
        out.push_back(std::move(p));
        rem.swap(keep);
    }
    return out;
}

double tile_cost(const GatePass& p, Arith ar) { return kPassBase[int(ar)] + p.inside; }

double scheduled_cost(const std::vector<Op>& ops, int n, Arith ar) {
    double t = 0.0;
    for (const GatePass& p : schedule_passes(ops, n, ar)) t += p.local ? std::min(p.alone, tile_cost(p, ar)) : p.alone;
    return t;
}

void launch_gate_pass(const GatePass& p, const std::vector<Op>& ops, void* psi, int n, Arith ar, bool ieee_in,
                      bool ieee_out, cudaStream_t st) {
    std::vector<const Op*> list;
    for (size_t i : p.ops) list.push_back(&ops[i]);
    const int k = int(list.size());
    switch (ar) {
        case Arith::F32: launch_pass_p<NativeArith<float>>(list.data(), k, p.data, p.local, psi, n, false, false, st); break;
        case Arith::F64: launch_pass_p<NativeArith<double>>(list.data(), k, p.data, p.local, psi, n, false, false, st); break;
        case Arith::DF: launch_pass_p<DFArith>(list.data(), k, p.data, p.local, psi, n, ieee_in, ieee_out, st); break;
    }
}

}  // namespace qs
