// Batched execution of many small parametric circuits in one persistent kernel launch,
// replayed from a CUDA graph: for every (circuit, observable) pair the energy
// E = <psi|H|psi> and the adjoint gradient dE/dtheta (reverse sweep of Sec. 4.4 parametric
// circuits, rotation convention exp(+i theta P / 2) of the paper's gate table), complex64
// storage; gradient partials are FP32 within a warp (at most 32 x 32 products) and FP64 across
// warps and chunks; the energy is a compensated (double-float) sum.
//
// Layout of the work:
//  * One CTA of 512 threads per SM claims work through atomic counters, longest first (the host
//    sorts by estimated cost): chunks of the circuits wider than 13 qubits level by level, with a
//    bounded grid barrier between levels, whole narrower circuits on groups of 1..16 warps.
//  * A circuit's gates are split on the host into passes. Each pass owns a window of at most
//    13 "local" qubits and holds gates acting only inside it; a gate joins the earliest pass
//    after every pass that touched its qubits and that still has room, so the passes applied in
//    order reproduce the circuit (gates outside a window commute with it). A pass is applied to
//    the state one chunk of 2^13 amplitudes at a time (the chunk fixes the other qubits), each
//    chunk staged in shared memory, so a whole pass costs one read and one write of the state.
//  * n <= 13: the whole state (and lambda) stays in shared memory for the entire circuit.
//  * A thread holds 16 amplitudes of psi (and of lambda) in registers for a stage. Z and CZ gates between
//    two others are one sign per amplitude; a rotation is one body (gradient chain, both
//    un-applications, the warp sum of the rotation before it) chosen by one branch, its two real
//    products per part in packed FP32 pairs. The order of the roundings is the circuit's.
//  * What bounds it: instruction issue (about 42 % of the slots, 16 warps per SM at 128 registers) and
//    the stage barriers; 1100 instructions per amplitude and layer at 18 qubits, a third of them FP32.
//    The next chunk's claim, look-ups and L2 prefetch run beside the current one's gates.
//    512 circuits of 8..20 qubits: 64.0 ms with a loop over separate gates (per-register phase signs,
//    one pass of negations per CZ, three branches per rotation), 48.0 ms with merged signs, packed
//    pairs and uniform signs, 47.0 ms with one body per rotation and the claim ahead. Merging the RZ
//    of a layer into one factor per amplitude measured 40.0 ms but changes the rounding of every
//    amplitude in FP32; it is not used.
//  * Forward sweep; lambda = H psi and E = Re <psi|lambda>; reverse sweep over passes and gates:
//    at a rotation exp(i theta P/2) the gradient is -Im <lambda|P|psi>, then the gate is
//    un-applied from psi and lambda.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <numeric>

#include "qsim_arith.cuh"

namespace qs {

namespace {

constexpr int kBT = 512;               // threads per CTA: 16 warps
constexpr int kWarps = kBT / 32;
constexpr int kLocal = 13;             // qubits per chunk
constexpr int kChunk = 1 << kLocal;    // 16 warps x 32 lanes x 16 registers
constexpr int kRegBits = 4;
constexpr int kRegs = 1 << kRegBits;
constexpr int kMaxStageRows = 32;   // gradient rows (sums per warp) of a stage
constexpr int kClasses = 5;            // groups of 16, 8, 4, 2, 1 warps
// a chunked pass's records kept in shared memory (larger passes read theirs from global memory)
constexpr int kUnitOps = 512, kUnitStages = 64, kUnitSigns = 64;
constexpr int kMaxBatchQubits = 24;

enum BKind : uint8_t { BK_RX = 0, BK_RY = 1, BK_RZ = 2, BK_CZ = 3, BK_CNOT = 4, BK_H = 5, BK_X = 6, BK_Y = 7, BK_Z = 8, BK_SIGN = 9 };

// one gate of a circuit before planning (host)
struct BGate {
    uint8_t kind;
    uint8_t a;      // target qubit (then the local bit of its pass)
    uint8_t b;      // second qubit (CZ) or control (CNOT)
    int32_t grad;   // gradient index (parametric rotations), -1 otherwise
};
constexpr uint8_t kNoReg = 0xff;

// one step of a stage: a rotation or fixed gate, or a run of sign gates (Z, CZ)
struct __align__(16) BOp {
    float2 cs;      // cos, sin of theta/2 (rotations; written before every run); sign run: its index (bits of x)
    uint8_t kind;
    uint8_t j;      // register bit of the target, or kNoReg (RZ)
    uint8_t b;      // RZ: local bit of the target; CNOT: of the control
    uint8_t jb;     // CNOT: register bit of the control, or kNoReg
    int16_t ref;    // rotations: gradient row of the stage (-1: none)
    uint8_t code;   // what the stage bodies branch on: kCode*
    uint8_t pad;
};
// rotations: their axis and register bit, one body each (RZ outside the registers: bit 4)
constexpr int kCodeRX = 0, kCodeRY = 4, kCodeRZ = 8, kCodeFixed = 13, kCodeSign = 14, kCodeGrad = 16;

// The signs of a run of Z and CZ gates: amplitude x of a thread (register index r, other local bits
// `base`) is negated where the parity of its Z bits and CZ pairs is odd.
struct BSign {
    uint32_t nbr[4];    // CZ partners of register bit j among the other bits
    uint32_t zbase;     // Z bits outside the registers
    uint32_t pat;       // sign of register index r from Z and CZ within the register bits, bit r
    int32_t cz0, ncz;   // CZ pairs on the other bits, grouped by distance
};
struct BCz {
    uint32_t shift, mask;  // pairs (a, a + shift), bit a set
};

// gates whose non-diagonal actions stay inside the register sub-cube spanned by act[] (register bit j
// is local bit act[j]; diagonal gates act on any bit)
struct BStage {
    int32_t o0, o1;     // steps
    int32_t p0, np;     // gradient outputs: parameter of each row
    uint8_t act[4];
    uint8_t sorted[4];  // act, ascending
};

struct BPass {
    int32_t s0, s1;               // stage range
    int32_t o0, o1, g0, g1;       // its steps and sign runs
    uint32_t tab_lo[128];         // local index bits 0..6 -> address bits
    uint32_t tab_hi[64];          // local index bits 7..12 -> address bits
    uint32_t nonlocal;            // qubits outside the window (fixed per chunk)
    int32_t nlocal;
};

struct BTerm {
    uint32_t xmask, zmask;
    double coef;
    int32_t nY, pad;
};

struct BItem {
    int32_t n;
    int32_t p0, p1;               // pass range
    int32_t t0, t1;               // observable term range
    int32_t angle0;               // first angle slot
    int32_t grad0, ngrad;         // gradient outputs
};

enum LevelKind : int32_t { LV_FWD = 0, LV_LAMBDA = 1, LV_REV = 2, LV_FINAL = 3 };
struct LevelEntry {
    int32_t item;
    int32_t pass;                 // pass index (forward / reverse levels)
    int32_t unit0;                // first unit of this entry within the level
    int32_t kind;
    uint64_t ws;                  // psi buffer of the item (amplitudes; lambda follows)
    int32_t n, first;             // first: a forward pass that starts from |0...0>
};
constexpr long long kBarrierSpinLimit = 1ll << 25;  // x 256 ns sleeps: ~10 s
// test hooks of the grid barrier (kernel arguments): polls before a wait gives up, and CTA 0
// holding back its arrival at the first barrier
std::atomic<long long> g_batch_polls{kBarrierSpinLimit};
std::atomic<int> g_batch_hold{0};

struct BatchDev {
    const BItem* items;
    const int32_t* order;         // resident items grouped by class, longest first within a class
    const BPass* passes;
    const BStage* stages;
    const BOp* ops;
    const BSign* signs;
    const BCz* czs;
    const int32_t* params;
    const BTerm* terms;
    float2* ws;                   // psi and lambda of every circuit wider than the window
    double* energy;
    double* grad;
    double* part_e;               // per wide item: energy partial per chunk
    const int64_t* part_e_off;
    double* part_g;               // per wide item: gradient partial per (parameter, chunk)
    const int64_t* part_g_off;
    const LevelEntry* lev_entries;
    const int32_t* lev_units;     // units per level
    const int32_t* lev_pair0;     // level -> first element of lev_pairs
    const int32_t* lev_pairs;     // entry of units 2 i and 2 i + 1 of a level (an entry has an even
                                  // number of units; the last level one per entry, see kind)
    int32_t nlevels;
    unsigned int* counters;       // kClasses resident counters, then one per level
    unsigned int* bar_count;
    unsigned int* bar_gen;
    int* err;
    long long barrier_polls;      // polls of a grid-barrier wait before it gives up
    int hold_cta;                 // test hook: CTA 0 does not arrive at the first grid barrier
    int32_t cls_begin[kClasses + 1];
};

// group barrier: the CTA, a named barrier over the group's warps, or the warp
__device__ __forceinline__ void gbar(int G, int w0) {
    if (G == kWarps) {
        __syncthreads();
    } else if (G == 1) {
        __syncwarp();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(1 + w0), "r"(G * 32) : "memory");
    }
}

// shared-memory position of local index l: the low four bits are XOR-folded with the higher
// ones so that lanes spread over the banks whichever bits are in registers
__device__ __forceinline__ uint32_t swz(uint32_t l) { return l ^ ((l >> 4) & 15u) ^ ((l >> 8) & 15u); }

__device__ __forceinline__ uint32_t chunk_base(uint32_t nonlocal, uint32_t c) {
    uint32_t r = 0, m = nonlocal;
    while (m) {
        const uint32_t bit = m & (0u - m);
        if (c & 1u) r |= bit;
        c >>= 1;
        m ^= bit;
    }
    return r;
}

// Chunk transfers between global memory and the shared-memory slice (the whole CTA: 512 threads x 16
// amplitudes, local index tg + 512 j). Local bits 0..8 are the thread's, 9..12 are j's, so an address
// is the thread's part OR j's masks, and a shared-memory position (swz is XOR-linear) the thread's
// XOR a constant.
struct ChunkMap {
    uint32_t off, hm[4], sw;
    __device__ __forceinline__ ChunkMap(const BPass& P, uint32_t base, int tg) {
        off = base | P.tab_lo[tg & 127] | P.tab_hi[tg >> 7];
#pragma unroll
        for (int k = 0; k < 4; k++) hm[k] = P.tab_hi[4 << k];
        sw = swz(uint32_t(tg));
    }
    __device__ __forceinline__ uint32_t addr(int j) const {
        uint32_t o = off;
#pragma unroll
        for (int k = 0; k < 4; k++)
            if ((j >> k) & 1) o |= hm[k];
        return o;
    }
    __device__ __forceinline__ uint32_t pos(int j) const { return sw ^ uint32_t((j << 9) ^ ((2 * j) & 15)); }
};
// every load is issued before the first store
template <bool kBoth>
__device__ __noinline__ void chunk_load(const ChunkMap m, const float2* __restrict__ g, const float2* __restrict__ h,
                                           float2* s, float2* t) {
    float2 v[kRegs], u[kRegs];
#pragma unroll
    for (int j = 0; j < kRegs; j++) v[j] = __ldcg(g + m.addr(j));
    if (kBoth) {
#pragma unroll
        for (int j = 0; j < kRegs; j++) u[j] = __ldcg(h + m.addr(j));
    }
#pragma unroll
    for (int j = 0; j < kRegs; j++) s[m.pos(j)] = v[j];
    if (kBoth) {
#pragma unroll
        for (int j = 0; j < kRegs; j++) t[m.pos(j)] = u[j];
    }
}
__device__ __noinline__ void chunk_store(const ChunkMap m, float2* __restrict__ g, const float2* s) {
#pragma unroll
    for (int j = 0; j < kRegs; j++) __stcg(g + m.addr(j), s[m.pos(j)]);
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// |0...0> restricted to a chunk: amplitude 1 at local index 0 of the chunk with base 0
__device__ __forceinline__ void sp_init(float2* s, uint32_t l, uint32_t base) {
    s[l ^ ((l >> 4) & 15u) ^ ((l >> 8) & 15u)] = make_float2((base == 0 && l == 0) ? 1.f : 0.f, 0.f);
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}

// Rotations on register bit J. The two parts of an amplitude share the real factors, so the updates
// run on packed FP32 pairs (each lane rounds as the scalar instruction).
// RY = [[c, s], [-s, c]]
template <int J>
__device__ __forceinline__ void pairs_ry(float2 (&v)[kRegs], float c, float sn) {
    const float2 c2 = make_float2(c, c), s2 = make_float2(sn, sn), m2 = make_float2(-sn, -sn);
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        if ((r >> J) & 1) continue;
        const int r1 = r | (1 << J);
        const float2 u = v[r], w = v[r1];
        v[r] = __ffma2_rn(c2, u, __fmul2_rn(s2, w));
        v[r1] = __ffma2_rn(c2, w, __fmul2_rn(m2, u));
    }
}
// RX = [[c, i s], [i s, c]]
template <int J>
__device__ __forceinline__ void pairs_rx(float2 (&v)[kRegs], float c, float sn) {
    const float2 c2 = make_float2(c, c), s2 = make_float2(-sn, sn);
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        if ((r >> J) & 1) continue;
        const int r1 = r | (1 << J);
        const float2 u = v[r], w = v[r1];
        v[r] = __ffma2_rn(c2, u, __fmul2_rn(s2, make_float2(w.y, w.x)));
        v[r1] = __ffma2_rn(c2, w, __fmul2_rn(s2, make_float2(u.y, u.x)));
    }
}
// H, X, Y (their own adjoints)
template <int J>
__device__ __forceinline__ void pairs_fixed(float2 (&v)[kRegs], uint8_t kind) {
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        if ((r >> J) & 1) continue;
        const int r1 = r | (1 << J);
        const float2 u = v[r], w = v[r1];
        if (kind == BK_H) {
            const float h = 0.70710678118654752f;
            v[r] = make_float2(fmaf(h, w.x, h * u.x), fmaf(h, w.y, h * u.y));
            v[r1] = make_float2(fmaf(-h, w.x, h * u.x), fmaf(-h, w.y, h * u.y));
        } else if (kind == BK_X) {
            v[r] = w;
            v[r1] = u;
        } else {  // Y = [[0, -i], [i, 0]]
            v[r] = make_float2(w.y, -w.x);
            v[r1] = make_float2(-u.y, u.x);
        }
    }
}
template <int J>
__device__ __forceinline__ void pairs_cnot(float2 (&v)[kRegs], uint32_t cmask) {
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        if ((r >> J) & 1) continue;
        const int r1 = r | (1 << J);
        if ((cmask >> r) & 1u) {
            const float2 u = v[r];
            v[r] = v[r1];
            v[r1] = u;
        }
    }
}
template <int J>
__device__ __forceinline__ void pairs_kind(float2 (&v)[kRegs], const BOp& o, uint32_t cmask) {
    if (o.kind == BK_CNOT) pairs_cnot<J>(v, cmask);
    else pairs_fixed<J>(v, o.kind);
}

// register indices with register bit j set
__device__ __forceinline__ uint32_t reg_pattern(int j) {
    return j == 0 ? 0xAAAAu : j == 1 ? 0xCCCCu : j == 2 ? 0xF0F0u : 0xFF00u;
}

// H, X, Y and CNOT (their own adjoints)
__device__ __forceinline__ void apply_fixed(float2 (&v)[kRegs], uint32_t base, const BOp& o) {
    uint32_t cmask = 0;
    if (o.kind == BK_CNOT) cmask = o.jb != kNoReg ? reg_pattern(o.jb) : ((base >> o.b) & 1u) ? 0xFFFFu : 0u;
    switch (o.j) {
        case 0: pairs_kind<0>(v, o, cmask); break;
        case 1: pairs_kind<1>(v, o, cmask); break;
        case 2: pairs_kind<2>(v, o, cmask); break;
        default: pairs_kind<3>(v, o, cmask); break;
    }
}

// RZ on register bit J (diag(c + i s, c - i s); the adjoint has -s) or, J == kRegBits, on a bit that
// is the same for all of the thread's registers (s signed by it)
template <int J>
__device__ __forceinline__ void phases_rz(float2 (&v)[kRegs], float c, float sn) {
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        const float s = (J < kRegBits && ((r >> J) & 1)) ? -sn : sn;
        v[r] = cmulf(make_float2(c, s), v[r]);
    }
}
// bit r: the sign of register index r under a run of sign gates
__device__ __forceinline__ uint32_t run_signs(const BatchDev& B, const BSign& D, uint32_t base) {
    uint32_t par = __popc(base & D.zbase);
    for (int k = 0; k < D.ncz; k++) {
        const BCz z = B.czs[D.cz0 + k];
        par ^= __popc(base & (base >> z.shift) & z.mask);
    }
    uint32_t m = D.pat ^ ((par & 1u) ? 0xFFFFu : 0u);
#pragma unroll
    for (int j = 0; j < kRegBits; j++) m ^= (__popc(base & D.nbr[j]) & 1) ? reg_pattern(j) : 0u;
    return m;
}
__device__ __forceinline__ float2 flip_if(float2 v, uint32_t sign, int r) {
    const uint32_t m = (sign << (31 - r)) & 0x80000000u;
    return make_float2(__uint_as_float(__float_as_uint(v.x) ^ m), __uint_as_float(__float_as_uint(v.y) ^ m));
}

// Im sum conj(lam) (P psi) over this thread's registers, P the axis of rotation o. The thread's
// partial (at most 32 products of complex64 data) is an FP32 FMA chain; the sums across warps and
// chunks are FP64.
template <int J>
__device__ __forceinline__ float grad_pairs(const float2 (&p)[kRegs], const float2 (&l)[kRegs], uint8_t kind) {
    float im = 0.f;
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        if ((r >> J) & 1) continue;
        const int r1 = r | (1 << J);
        const float2 a = p[r], b = p[r1], la = l[r], lb = l[r1];
        float2 p0, p1;  // X -> (b, a); Y -> (-i b, i a)
        if (kind == BK_RX) { p0 = b; p1 = a; }
        else { p0 = make_float2(b.y, -b.x); p1 = make_float2(-a.y, a.x); }
        im = fmaf(la.x, p0.y, im);
        im = fmaf(-la.y, p0.x, im);
        im = fmaf(lb.x, p1.y, im);
        im = fmaf(-lb.y, p1.x, im);
    }
    return im;
}
// Z on register bit J; J == kRegBits: without the sign, which is the same for all registers
template <int J>
__device__ __forceinline__ float grad_z(const float2 (&p)[kRegs], const float2 (&l)[kRegs]) {
    float im = 0.f;
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        const bool neg = J < kRegBits && ((r >> J) & 1);
        im = fmaf(neg ? -l[r].x : l[r].x, p[r].y, im);
        im = fmaf(neg ? l[r].y : -l[r].y, p[r].x, im);
    }
    return im;
}
// One rotation (its code without the gradient flag): un-applied or applied
template <int kCode>
__device__ __forceinline__ void rotate(float2 (&v)[kRegs], float c, float sn, uint32_t bit) {
    if constexpr (kCode < kCodeRY) pairs_rx<kCode>(v, c, sn);
    else if constexpr (kCode < kCodeRZ) pairs_ry<kCode - kCodeRY>(v, c, sn);
    else if constexpr (kCode < kCodeRZ + kRegBits) phases_rz<kCode - kCodeRZ>(v, c, sn);
    else phases_rz<kRegBits>(v, c, bit ? -sn : sn);
}
template <int kCode>
__device__ __forceinline__ float rotation_grad(const float2 (&p)[kRegs], const float2 (&l)[kRegs], uint32_t bit) {
    if constexpr (kCode < kCodeRY) return grad_pairs<kCode>(p, l, BK_RX);
    else if constexpr (kCode < kCodeRZ) return grad_pairs<kCode - kCodeRY>(p, l, BK_RY);
    else if constexpr (kCode < kCodeRZ + kRegBits) return grad_z<kCode - kCodeRZ>(p, l);
    else {
        const float g = grad_z<kRegBits>(p, l);
        return bit ? -g : g;
    }
}

// Thread tg of a stage holds the 16 amplitudes of the register sub-cube at `base` (its bits spread
// over the local bits outside act, ascending). The shared-memory positions are XOR-linear in the
// index: one XOR per register from the stage's four masks (in bytes).
struct StageMap {
    uint32_t base, a0, am[kRegBits];
    __device__ __forceinline__ StageMap(const BStage& S, int tg) {
        uint32_t t = uint32_t(tg);
#pragma unroll
        for (int j = 0; j < kRegBits; j++) {
            const uint32_t lo = t & ((1u << S.sorted[j]) - 1u);
            t = ((t ^ lo) << 1) | lo;
            am[j] = swz(1u << S.act[j]) * uint32_t(sizeof(float2));
        }
        base = t;
        a0 = swz(t) * uint32_t(sizeof(float2));
    }
    __device__ __forceinline__ float2* at(float2* s, int r) const {
        uint32_t o = a0;
#pragma unroll
        for (int j = 0; j < kRegBits; j++)
            if ((r >> j) & 1) o ^= am[j];
        return reinterpret_cast<float2*>(reinterpret_cast<unsigned char*>(s) + o);
    }
};

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// ---------------------------------------------------------------- stage bodies
// where a pass's steps are read from: shared memory for a chunked pass that fits, else global
struct StepSource {
    const BOp* ops;
    const BSign* signs;
};
// forward: registers <- slice, gates, slice <- registers
__device__ __forceinline__ void stage_forward(const BatchDev& B, const BStage& S, StepSource src, int tg, int T,
                                              float2* sp) {
    if (tg >= T) return;
    const StageMap m(S, tg);
    float2 v[kRegs];
#pragma unroll
    for (int r = 0; r < kRegs; r++) v[r] = *m.at(sp, r);
    BOp o = src.ops[S.o0];
    for (int i = S.o0; i < S.o1; i++) {
        const BOp next = i + 1 < S.o1 ? src.ops[i + 1] : o;  // prefetch
        const float c = o.cs.x, sn = o.cs.y;
        const uint32_t bit = (m.base >> (o.b & 31)) & 1u;
        switch (o.code & 15) {
#define QS_ROT(k) \
    case k: rotate<k>(v, c, sn, bit); break;
            QS_ROT(0) QS_ROT(1) QS_ROT(2) QS_ROT(3) QS_ROT(4) QS_ROT(5) QS_ROT(6) QS_ROT(7)
            QS_ROT(8) QS_ROT(9) QS_ROT(10) QS_ROT(11) QS_ROT(12)
#undef QS_ROT
            case kCodeSign: {
                const uint32_t sign = run_signs(B, src.signs[__float_as_int(c)], m.base);
#pragma unroll
                for (int r = 0; r < kRegs; r++) v[r] = flip_if(v[r], sign, r);
                break;
            }
            default: apply_fixed(v, m.base, o); break;
        }
        o = next;
    }
#pragma unroll
    for (int r = 0; r < kRegs; r++) *m.at(sp, r) = v[r];
}

// reverse: gradient rows of the stage into red[row][warp], un-apply from psi and lambda. Every lane
// reaches the warp sums; lanes beyond T (never with kFull) hold zeros and store nothing.
template <bool kFull>
__device__ __forceinline__ void stage_reverse(const BatchDev& B, const BStage& S, StepSource src, int tg, int T,
                                              float2* sp, float2* sl, float (*red)[kWarps], int warp, int lane) {
    const bool active = kFull || tg < T;
    const StageMap m(S, tg);
    float2 v[kRegs], u[kRegs];
#pragma unroll
    for (int r = 0; r < kRegs; r++) {
        v[r] = active ? *m.at(sp, r) : make_float2(0.f, 0.f);
        u[r] = active ? *m.at(sl, r) : make_float2(0.f, 0.f);
    }
    // One body per rotation: its gradient's FMA chain, both un-applications and the warp sum of the
    // rotation before it (held back one step) are independent, so that their latencies overlap.
    float held = 0.f;
    int held_row = -1;
    BOp o = src.ops[S.o1 - 1];
    for (int i = S.o1 - 1; i >= S.o0; i--) {
        const BOp next = i > S.o0 ? src.ops[i - 1] : o;  // prefetch
        const float c = o.cs.x, sn = -o.cs.y;
        const uint32_t bit = (m.base >> (o.b & 31)) & 1u;
        switch (o.code) {
#define QS_ROT(k)                                              \
    case k:                                                    \
        rotate<k>(v, c, sn, bit);                              \
        rotate<k>(u, c, sn, bit);                              \
        break;                                                 \
    case kCodeGrad + k: {                                      \
        const float sum = warp_sum_f(held);                    \
        held = rotation_grad<k>(v, u, bit);                    \
        rotate<k>(v, c, sn, bit);                              \
        rotate<k>(u, c, sn, bit);                              \
        if (lane == 0 && held_row >= 0) red[held_row][warp] = sum; \
        held_row = o.ref;                                      \
        break;                                                 \
    }
            QS_ROT(0) QS_ROT(1) QS_ROT(2) QS_ROT(3) QS_ROT(4) QS_ROT(5) QS_ROT(6) QS_ROT(7)
            QS_ROT(8) QS_ROT(9) QS_ROT(10) QS_ROT(11) QS_ROT(12)
#undef QS_ROT
            case kCodeSign: {
                const uint32_t sign = run_signs(B, src.signs[__float_as_int(c)], m.base);
#pragma unroll
                for (int r = 0; r < kRegs; r++) {
                    v[r] = flip_if(v[r], sign, r);
                    u[r] = flip_if(u[r], sign, r);
                }
                break;
            }
            default:
                apply_fixed(v, m.base, o);
                apply_fixed(u, m.base, o);
                break;
        }
        o = next;
    }
    if (held_row >= 0) {
        const float sum = warp_sum_f(held);
        if (lane == 0) red[held_row][warp] = sum;
    }
    if (active) {
#pragma unroll
        for (int r = 0; r < kRegs; r++) {
            *m.at(sp, r) = v[r];
            *m.at(sl, r) = u[r];
        }
    }
}

// after the stage barrier: row k's sum over the group's G warps (FP64, a fixed tree) by warp k mod G of
// the group, dE/dtheta = -Im <lambda|P|psi> added to out[stride * parameter] (each address belongs to
// this group; a reduction without a return value does not stall the warp)
__device__ __forceinline__ void row_sums(const int32_t* params, int np, const float (*red)[kWarps], int w0, int G,
                                         int warp, int lane, double* out, size_t stride) {
    for (int k = warp - w0; k < np; k += G) {
        double v = lane < G ? double(red[k][w0 + lane]) : 0.0;
        for (int o = G / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) atomicAdd(out + stride * size_t(params[k]), -v);
    }
}

// lambda_y = sum_t coef i^{#Y} s(y ^ f) psi_{y ^ f} for y in [y0, y1) (stride nthr), and this
// thread's share of Re <psi|lambda>; src/dst are shared slices (resident) or global buffers
template <bool RES>
__device__ __forceinline__ double lambda_range(const BatchDev& B, const BItem& it, const float2* src, float2* dst,
                                               uint32_t y0, uint32_t y1, int tg, int nthr) {
    DFAcc e;
    df_zero(e);
    const int nt = it.t1 - it.t0;
    for (uint32_t y = y0 + tg; y < y1; y += nthr) {
        float2 s4[4];
#pragma unroll
        for (int t = 0; t < 4; t++)
            if (t < nt) {
                const uint32_t y2 = y ^ B.terms[it.t0 + t].xmask;
                s4[t] = RES ? src[swz(y2)] : src[y2];
            }
        const float2 ps = RES ? src[swz(y)] : src[y];
        float re = 0.f, im = 0.f;  // lambda is stored as complex64
        for (int t = 0; t < nt; t++) {
            const BTerm Tm = B.terms[it.t0 + t];
            const uint32_t y2 = y ^ Tm.xmask;
            float2 v = t < 4 ? s4[min(t, 3)] : (RES ? src[swz(y2)] : src[y2]);
            v = mul_ipow(v, Tm.nY + 2 * (__popc(y2 & Tm.zmask) & 1));
            re = fmaf(float(Tm.coef), v.x, re);
            im = fmaf(float(Tm.coef), v.y, im);
        }
        const float2 lam = make_float2(re, im);
        if (RES) dst[swz(y)] = lam; else dst[y] = lam;
        df_add_prod(e, ps.x, lam.x);
        df_add_prod(e, ps.y, lam.y);
    }
    return df_value(e);
}

// grid-wide barrier with a bounded wait (all CTAs are co-resident: cooperative launch). On
// timeout it sets the error flag and returns false; every caller then leaves the kernel. A CTA
// told to hold back (a test of the timeout) waits without arriving, so that every wait runs out.
__device__ bool grid_barrier(unsigned int* count, unsigned int* gen, int* err, long long polls, bool hold) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        volatile unsigned int* vgen = gen;
        const unsigned int g = *vgen;
        __threadfence();
        int ok = 1;
        if (!hold && atomicAdd(count, 1u) == gridDim.x - 1) {
            *count = 0;
            __threadfence();
            atomicAdd(gen, 1u);
        } else {
            long long spins = 0;
            while (*vgen == g) {
                if (++spins > polls || *(volatile int*)err) {
                    atomicExch(err, 1);
                    ok = 0;
                    break;
                }
                __nanosleep(256);
            }
        }
        __threadfence();
        s_ok = ok && !*(volatile int*)err;
    }
    __syncthreads();
    return s_ok != 0;
}

// a claimed unit of a level (kind < 0: none left)
struct BUnit {
    int32_t kind, item, pass, n, first;
    uint32_t c;
    uint64_t ws;
};
__device__ __noinline__ void claim_unit(const BatchDev& B, int lv, int total, BUnit& out) {
    const int u = int(atomicAdd(&B.counters[kClasses + lv], 1u));
    if (u >= total) {
        out.kind = -1;
        return;
    }
    const int pair = B.lev_pair0[lv];
    const LevelEntry E = B.lev_entries[pair < 0 ? ~pair + u : B.lev_pairs[pair + (u >> 1)]];
    out.kind = E.kind;
    out.item = E.item;
    out.pass = E.pass;
    out.n = E.n;
    out.first = E.first;
    out.c = uint32_t(u - E.unit0);
    out.ws = E.ws;
}
// a chunk that the next unit reads, into L2: one 128-byte line (16 amplitudes) per thread and buffer
__device__ __forceinline__ void prefetch_unit(const BatchDev& B, const BUnit& U, int tg) {
    if (U.kind < 0 || U.first) return;
    const BPass& P = B.passes[U.pass];
    const uint32_t l = uint32_t(tg) * 16u;
    const float2* p = B.ws + U.ws + (chunk_base(P.nonlocal, U.c) | P.tab_lo[l & 127] | P.tab_hi[l >> 7]);
    prefetch_l2(p);
    if (U.kind == LV_REV) prefetch_l2(p + (uint64_t(1) << U.n));
}
__device__ __forceinline__ void copy_words(void* dst, const void* src, int words, int tg) {
    for (int i = tg; i < words; i += kBT) static_cast<uint32_t*>(dst)[i] = static_cast<const uint32_t*>(src)[i];
}

__global__ void __launch_bounds__(kBT, 1) k_batch(const BatchDev B) {
    extern __shared__ __align__(16) unsigned char smem[];
    float2* smem_p = reinterpret_cast<float2*>(smem);
    float2* smem_l = smem_p + kChunk;
    __shared__ float red[2][kMaxStageRows][kWarps];  // gradient partials per stage parity
    __shared__ double redE[kWarps];
    __shared__ int s_claim[kWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ BUnit s_unit[2];
    __shared__ __align__(16) BOp s_ops[kUnitOps];
    __shared__ BStage s_stages[kUnitStages];
    __shared__ BSign s_signs[kUnitSigns];
    int parity = 0;
    bool first_barrier = true;

    // ================= circuits wider than the window: level-synchronous over the grid
    for (int lv = 0; lv < B.nlevels; lv++) {
        const int total = B.lev_units[lv];
        // units are claimed one ahead: the claim and its look-ups run while the current unit's chunk is
        // on its way from memory, and the next chunk is fetched into L2 during the current one's gates
        if (threadIdx.x == 0) claim_unit(B, lv, total, s_unit[0]);
        __syncthreads();
        for (int cur = 0; s_unit[cur].kind >= 0; cur ^= 1) {
            const BUnit E = s_unit[cur];
            const uint32_t c = E.c;
            const uint32_t nch = 1u << (E.n - kLocal);
            float2* gpsi = B.ws + E.ws;
            float2* glam = gpsi + (uint64_t(1) << E.n);
            const int tg = threadIdx.x;
            if (E.kind == LV_FWD || E.kind == LV_REV) {
                const BPass& P = B.passes[E.pass];
                const ChunkMap m(P, chunk_base(P.nonlocal, c), tg);
                const int ns = P.s1 - P.s0, no = P.o1 - P.o0, ng = P.g1 - P.g0;
                const bool fits = ns <= kUnitStages && no <= kUnitOps && ng <= kUnitSigns;
                if (fits) {  // the pass's records, on their way beside the chunk
                    copy_words(s_stages, B.stages + P.s0, ns * int(sizeof(BStage) / 4), tg);
                    copy_words(s_ops, B.ops + P.o0, no * int(sizeof(BOp) / 4), tg);
                    copy_words(s_signs, B.signs + P.g0, ng * int(sizeof(BSign) / 4), tg);
                }
                const BStage* stages = fits ? s_stages - P.s0 : B.stages;
                const StepSource src{fits ? s_ops - P.o0 : B.ops, fits ? s_signs - P.g0 : B.signs};
                if (tg == 0) claim_unit(B, lv, total, s_unit[cur ^ 1]);
                if (E.kind == LV_FWD) {
                    if (E.first) {
                        const uint32_t base = chunk_base(P.nonlocal, c);
                        for (uint32_t l = tg; l < kChunk; l += kBT) sp_init(smem_p, l, base);
                    } else {
                        chunk_load<false>(m, gpsi, nullptr, smem_p, nullptr);
                    }
                    __syncthreads();
                    prefetch_unit(B, s_unit[cur ^ 1], tg);
                    for (int s = P.s0; s < P.s1; s++) {
                        stage_forward(B, stages[s], src, tg, kBT, smem_p);
                        __syncthreads();
                    }
                    chunk_store(m, gpsi, smem_p);
                } else {
                    chunk_load<true>(m, gpsi, glam, smem_p, smem_l);
                    __syncthreads();
                    prefetch_unit(B, s_unit[cur ^ 1], tg);
                    double* pg = B.part_g + B.part_g_off[E.item] + c;
                    for (int s = P.s1 - 1; s >= P.s0; s--) {
                        const BStage S = stages[s];
                        stage_reverse<true>(B, S, src, tg, kBT, smem_p, smem_l, red[parity], warp, lane);
                        __syncthreads();
                        row_sums(B.params + S.p0, S.np, red[parity], 0, kWarps, warp, lane, pg, nch);
                        parity ^= 1;
                    }
                    chunk_store(m, gpsi, smem_p);
                    chunk_store(m, glam, smem_l);
                }
                __syncthreads();
            } else if (E.kind == LV_LAMBDA) {
                if (tg == 0) claim_unit(B, lv, total, s_unit[cur ^ 1]);
                const uint32_t y0 = c << kLocal;
                const double ew = warp_sum(lambda_range<false>(B, B.items[E.item], gpsi, glam, y0, y0 + kChunk, tg, kBT));
                if (lane == 0) redE[warp] = ew;
                __syncthreads();
                if (tg == 0) {
                    double e = 0.0;
                    for (int w = 0; w < kWarps; w++) e += redE[w];
                    B.part_e[B.part_e_off[E.item] + c] = e;
                }
                __syncthreads();
            } else {  // LV_FINAL: energy and gradients of the item, sums in chunk order
                const int item = E.item;
                const BItem it = B.items[item];
                if (tg == 0) {
                    claim_unit(B, lv, total, s_unit[cur ^ 1]);
                    double e = 0.0;
                    for (uint32_t k = 0; k < nch; k++) e += B.part_e[B.part_e_off[item] + k];
                    B.energy[item] = e;
                }
                const double* pg = B.part_g + B.part_g_off[item];
                for (int j = tg; j < it.ngrad; j += kBT) {
                    double gsum = 0.0;
                    for (uint32_t k = 0; k < nch; k++) gsum += pg[size_t(j) * nch + k];
                    B.grad[it.grad0 + j] = gsum;
                }
                __syncthreads();
            }
        }
        if (!grid_barrier(B.bar_count, B.bar_gen, B.err, B.barrier_polls, B.hold_cta && blockIdx.x == 0 && first_barrier))
            return;
        first_barrier = false;
    }

    // ================= circuits within the window: whole circuit per warp group, in shared memory
    for (int cls = 0; cls < kClasses; cls++) {
        const int G = kWarps >> cls;
        const int w0 = (warp / G) * G;
        const int tg = threadIdx.x - w0 * 32;
        const int nthr = G * 32;
        float2* sp = smem_p + w0 * 32 * kRegs;
        float2* sl = smem_l + w0 * 32 * kRegs;
        const int count = B.cls_begin[cls + 1] - B.cls_begin[cls];
        while (true) {
            if (tg == 0) s_claim[w0] = int(atomicAdd(&B.counters[cls], 1u));
            gbar(G, w0);
            const int k = s_claim[w0];
            gbar(G, w0);
            if (k >= count) break;
            const int item = B.order[B.cls_begin[cls] + k];
            const BItem it = B.items[item];
            const uint32_t size = 1u << it.n;
            const int T = int(size) / kRegs;
            for (int j = tg; j < it.ngrad; j += nthr) B.grad[it.grad0 + j] = 0.0;
            for (uint32_t l = tg; l < size; l += nthr) sp_init(sp, l, 0u);
            gbar(G, w0);
            const BPass& P = B.passes[it.p0];  // one pass holds the whole circuit
            for (int s = P.s0; s < P.s1; s++) {
                stage_forward(B, B.stages[s], StepSource{B.ops, B.signs}, tg, T, sp);
                gbar(G, w0);
            }
            {
                const double ew = warp_sum(lambda_range<true>(B, it, sp, sl, 0u, size, tg, nthr));
                if (lane == 0) redE[warp] = ew;
                gbar(G, w0);
                if (tg == 0) {
                    double E = 0.0;
                    for (int w = w0; w < w0 + G; w++) E += redE[w];
                    B.energy[item] = E;
                }
                gbar(G, w0);
            }
            for (int s = P.s1 - 1; s >= P.s0; s--) {
                const BStage S = B.stages[s];
                stage_reverse<false>(B, S, StepSource{B.ops, B.signs}, tg, T, sp, sl, red[parity], warp, lane);
                gbar(G, w0);
                row_sums(B.params + S.p0, S.np, red[parity], w0, G, warp, lane, B.grad + it.grad0, 1);
                parity ^= 1;
            }
        }
    }
}

// (cos, sin) of theta/2 of every angle slot into its step
__global__ void k_angles(const double* __restrict__ theta, const uint32_t* __restrict__ op, BOp* __restrict__ ops, int count) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        double s, c;
        sincos(0.5 * theta[i], &s, &c);
        ops[op[i]].cs = make_float2(float(c), float(s));
    }
}

}  // namespace

}  // namespace qs

// ------------------------------------------------------------------ host side
struct qs_batch {
    int count = 0;
    int total_grads = 0;
    int total_angles = 0;
    int max_n = 0;
    std::vector<qs::BItem> items;
    std::vector<int32_t> order;
    std::vector<qs::BPass> passes;
    std::vector<qs::BStage> stages;
    std::vector<qs::BOp> ops;
    std::vector<qs::BSign> signs;
    std::vector<qs::BCz> czs;
    std::vector<int32_t> params;
    std::vector<uint32_t> angle_op;     // angle slot -> the step it belongs to
    std::vector<qs::BTerm> terms;
    std::vector<int32_t> angle_param;   // angle slot -> parameter index of its circuit (or -1)
    std::vector<double> angle_fixed;    // angle slot -> fixed angle (when not parametric)
    std::vector<int32_t> angle_item;    // angle slot -> item
    std::vector<int32_t> param0;        // item -> first parameter in the caller's theta array
    std::vector<int32_t> grad_of_item;  // item -> grad0
    // circuits wider than the window: buffers and levels
    std::vector<uint64_t> ws_off;       // item -> psi offset (amplitudes)
    std::vector<int64_t> part_e_off, part_g_off;
    std::vector<qs::LevelEntry> lev_entries;
    std::vector<int32_t> lev_units, lev_pair0, lev_pairs;
    uint64_t ws_amps = 0;
    int64_t part_e_total = 0, part_g_total = 0;
    // device buffers
    void* d_items = nullptr;
    void* d_order = nullptr;
    void* d_passes = nullptr;
    void* d_stages = nullptr;
    void* d_ops = nullptr;
    void* d_signs = nullptr;
    void* d_angle_op = nullptr;
    void* d_czs = nullptr;
    void* d_params = nullptr;
    void* d_terms = nullptr;
    double* d_theta = nullptr;
    float2* d_ws = nullptr;
    double* d_part_e = nullptr;
    void* d_part_e_off = nullptr;
    double* d_part_g = nullptr;
    void* d_part_g_off = nullptr;
    void* d_lev_entries = nullptr;
    void* d_lev_pair0 = nullptr;
    void* d_lev_pairs = nullptr;
    void* d_lev_units = nullptr;
    unsigned int* d_bar = nullptr;    // count, generation
    int* d_err = nullptr;
    int* h_err = nullptr;             // pinned
    double* d_energy = nullptr;
    double* d_grad = nullptr;
    unsigned int* d_counter = nullptr;
    double* h_theta = nullptr;   // pinned
    double* h_energy = nullptr;  // pinned
    double* h_grad = nullptr;    // pinned
    int cls_begin[qs::kClasses + 1] = {};
    int grid = 0;
    size_t smem = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaStream_t graph_stream = nullptr;
    long long graph_polls = 0;   // wait-test settings the graph was captured with
    int graph_hold = 0;
    int device = 0;
};

namespace qs {
namespace {

// The gates of a pass (local bits, circuit order) as stages: a stage takes gates in order until their
// non-diagonal targets need a fifth register bit, its gradient rows run out or a parameter comes a
// second time. Z and CZ gates between two gates that are not diagonal become one run of signs at its
// end: negations are exact and commute with the phases among them.
void plan_stages(const std::vector<BGate>& gl, const std::vector<int32_t>& slot, int nl, qs_batch& b) {
    auto diagonal = [](const BGate& g) { return g.kind == BK_RZ || g.kind == BK_Z || g.kind == BK_CZ; };
    std::vector<int> cur, act, grads;
    auto close_stage = [&]() {
        if (cur.empty()) return;
        for (int q = 0; q < nl && int(act.size()) < kRegBits; q++)
            if (std::find(act.begin(), act.end(), q) == act.end()) act.push_back(q);
        BStage st;
        std::memset(&st, 0, sizeof(st));
        st.o0 = int(b.ops.size());
        st.p0 = int(b.params.size());
        for (int j = 0; j < kRegBits; j++) st.act[j] = st.sorted[j] = uint8_t(act[j]);
        std::sort(st.sorted, st.sorted + kRegBits);
        auto regpos = [&](int bit) {
            const auto f = std::find(act.begin(), act.end(), bit);
            return f == act.end() ? kNoReg : uint8_t(f - act.begin());
        };
        const uint32_t pat[kRegBits] = {0xAAAAu, 0xCCCCu, 0xF0F0u, 0xFF00u};
        BSign D;
        std::map<int, uint32_t> pairs;  // distance -> lower bits of the run's CZ pairs outside the registers
        bool open = false;
        auto close_run = [&]() {
            if (!open) return;
            D.cz0 = int(b.czs.size());
            for (const auto& pm : pairs)
                if (pm.second) b.czs.push_back(BCz{uint32_t(pm.first), pm.second});
            D.ncz = int(b.czs.size()) - D.cz0;
            pairs.clear();
            open = false;
            BOp o;
            std::memset(&o, 0, sizeof(o));
            o.kind = BK_SIGN;
            o.code = kCodeSign;
            o.ref = -1;
            const int32_t index = int32_t(b.signs.size());
            std::memcpy(&o.cs.x, &index, sizeof(index));
            b.signs.push_back(D);
            b.ops.push_back(o);
        };
        for (int i : cur) {
            const BGate& g = gl[i];
            const uint8_t ja = regpos(g.a);
            if (g.kind == BK_Z || g.kind == BK_CZ) {
                if (!open) std::memset(&D, 0, sizeof(D));
                open = true;
                if (g.kind == BK_Z) {
                    if (ja != kNoReg) D.pat ^= pat[ja];
                    else D.zbase ^= 1u << g.a;
                    continue;
                }
                const uint8_t jb = regpos(g.b);
                if (ja != kNoReg && jb != kNoReg) D.pat ^= pat[ja] & pat[jb];
                else if (ja != kNoReg) D.nbr[ja] ^= 1u << g.b;
                else if (jb != kNoReg) D.nbr[jb] ^= 1u << g.a;
                else pairs[std::abs(int(g.a) - int(g.b))] ^= 1u << std::min(g.a, g.b);
                continue;
            }
            if (g.kind != BK_RZ) close_run();
            BOp o;
            std::memset(&o, 0, sizeof(o));
            o.cs = make_float2(1.f, 0.f);
            o.kind = g.kind;
            o.j = ja;
            o.b = g.kind == BK_CNOT ? g.b : g.a;
            o.jb = g.kind == BK_CNOT ? regpos(g.b) : kNoReg;
            o.ref = -1;
            o.code = uint8_t(g.kind == BK_RX ? kCodeRX + ja : g.kind == BK_RY ? kCodeRY + ja
                             : g.kind == BK_RZ ? kCodeRZ + (ja == kNoReg ? kRegBits : ja) : kCodeFixed);
            if (g.grad >= 0) {
                o.ref = int16_t(int(b.params.size()) - st.p0);
                o.code |= kCodeGrad;
                b.params.push_back(g.grad);
            }
            if (slot[i] >= 0) b.angle_op[slot[i]] = uint32_t(b.ops.size());
            b.ops.push_back(o);
        }
        close_run();
        st.o1 = int(b.ops.size());
        st.np = int(b.params.size()) - st.p0;
        b.stages.push_back(st);
        cur.clear();
        act.clear();
        grads.clear();
    };
    for (size_t i = 0; i < gl.size(); i++) {
        const BGate& g = gl[i];
        const bool diag = diagonal(g);
        const bool have = diag || std::find(act.begin(), act.end(), int(g.a)) != act.end();
        const bool row = g.grad >= 0;
        if ((row && int(grads.size()) >= kMaxStageRows) || (!have && int(act.size()) >= kRegBits) ||
            (row && std::find(grads.begin(), grads.end(), g.grad) != grads.end()))
            close_stage();
        if (!diag && std::find(act.begin(), act.end(), int(g.a)) == act.end()) act.push_back(g.a);
        cur.push_back(int(i));
        if (row) grads.push_back(g.grad);
    }
    close_stage();
}

// split one circuit into passes over windows of <= kLocal qubits
void plan_passes(const qs_circuit& c, const std::vector<BGate>& gl, const std::vector<uint32_t>& gmask,
                 const std::vector<int32_t>& gslot,
                 qs_batch& b, BItem& it) {
    const int n = c.n;
    const int win = std::min(n, kLocal);
    struct P {
        uint32_t mask = 0;
        std::vector<int> gates;
    };
    std::vector<P> ps;
    std::vector<int> last(n, -1);
    const uint32_t low = (1u << std::min(5, win)) - 1u;  // keep the 5 lowest qubits local: 256-byte runs
    for (size_t i = 0; i < gl.size(); i++) {
        const uint32_t m = gmask[i];
        int dep = -1;
        for (int q = 0; q < n; q++)
            if ((m >> q) & 1) dep = std::max(dep, last[q]);
        int chosen = -1;
        for (int p = std::max(dep, 0); p < int(ps.size()); p++) {
            if (p < dep) continue;
            if (__builtin_popcount(ps[p].mask | m | low) <= win) {
                chosen = p;
                break;
            }
        }
        if (chosen < 0) {
            ps.emplace_back();
            chosen = int(ps.size()) - 1;
        }
        ps[chosen].mask |= m;
        ps[chosen].gates.push_back(int(i));
        for (int q = 0; q < n; q++)
            if ((m >> q) & 1) last[q] = chosen;
    }
    if (ps.empty()) ps.emplace_back();
    it.p0 = int(b.passes.size());
    for (auto& p : ps) {
        // window: the pass's qubits, the lowest qubits, then fill with the lowest unused ones
        uint32_t w = p.mask | low;
        for (int q = 0; q < n && __builtin_popcount(w) < win; q++) w |= 1u << q;
        std::vector<int> lq;
        for (int q = 0; q < n; q++)
            if ((w >> q) & 1) lq.push_back(q);
        BPass bp;
        std::memset(&bp, 0, sizeof(bp));
        bp.nlocal = int(lq.size());
        bp.nonlocal = ((n >= 32) ? 0xffffffffu : ((1u << n) - 1u)) & ~w;
        for (int l = 0; l < 128; l++) {
            uint32_t a = 0;
            for (int j = 0; j < 7 && j < int(lq.size()); j++)
                if ((l >> j) & 1) a |= 1u << lq[j];
            bp.tab_lo[l] = a;
        }
        for (int h = 0; h < 64; h++) {
            uint32_t a = 0;
            for (int j = 0; j < 6 && 7 + j < int(lq.size()); j++)
                if ((h >> j) & 1) a |= 1u << lq[7 + j];
            bp.tab_hi[h] = a;
        }
        auto local = [&](int q) { return uint8_t(std::find(lq.begin(), lq.end(), q) - lq.begin()); };
        std::vector<BGate> pg;
        std::vector<int32_t> ps;
        for (int gi : p.gates) {
            BGate g = gl[gi];
            g.a = local(g.a);
            if (g.kind == BK_CZ || g.kind == BK_CNOT) g.b = local(g.b);
            pg.push_back(g);
            ps.push_back(gslot[gi]);
        }
        bp.s0 = int(b.stages.size());
        bp.o0 = int(b.ops.size());
        bp.g0 = int(b.signs.size());
        plan_stages(pg, ps, int(lq.size()), b);
        bp.s1 = int(b.stages.size());
        bp.o1 = int(b.ops.size());
        bp.g1 = int(b.signs.size());
        b.passes.push_back(bp);
    }
    it.p1 = int(b.passes.size());
}

void free_batch(qs_batch* b) {
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    if (b->graph_stream) cudaStreamDestroy(b->graph_stream);
    void* dev[] = {b->d_items, b->d_order, b->d_passes, b->d_stages, b->d_ops, b->d_signs, b->d_angle_op, b->d_czs, b->d_params, b->d_terms,
                   b->d_theta, b->d_ws, b->d_part_e, b->d_part_e_off, b->d_part_g, b->d_part_g_off,
                   b->d_lev_entries, b->d_lev_pair0, b->d_lev_pairs, b->d_lev_units, b->d_bar, b->d_err, b->d_energy, b->d_grad,
                   b->d_counter};
    for (void* p : dev)
        if (p) dev_free(p);
    if (b->h_theta) host_free_pinned(b->h_theta);
    if (b->h_energy) host_free_pinned(b->h_energy);
    if (b->h_grad) host_free_pinned(b->h_grad);
    if (b->h_err) host_free_pinned(b->h_err);
}

template <typename T>
void upload(void** d, const std::vector<T>& h) {
    const size_t bytes = std::max<size_t>(1, h.size()) * sizeof(T);
    QS_TRY_CUDA(dev_malloc(d, bytes));
    if (!h.empty()) QS_TRY_CUDA(cudaMemcpy(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
}

// enqueue one batch evaluation on `st` (used directly and under graph capture)
void enqueue(qs_batch* b, cudaStream_t st) {
    QS_TRY_CUDA(cudaMemcpyAsync(b->d_theta, b->h_theta, sizeof(double) * std::max(1, b->total_angles),
                                cudaMemcpyHostToDevice, st));
    k_angles<<<std::max(1, std::min(1024, (b->total_angles + 255) / 256)), 256, 0, st>>>(
        b->d_theta, static_cast<const uint32_t*>(b->d_angle_op), static_cast<BOp*>(b->d_ops), b->total_angles);
    const int nlev = int(b->lev_units.size());
    QS_TRY_CUDA(cudaMemsetAsync(b->d_counter, 0, sizeof(unsigned int) * (kClasses + nlev), st));
    QS_TRY_CUDA(cudaMemsetAsync(b->d_bar, 0, sizeof(unsigned int) * 2, st));
    QS_TRY_CUDA(cudaMemsetAsync(b->d_err, 0, sizeof(int), st));
    if (b->part_g_total) QS_TRY_CUDA(cudaMemsetAsync(b->d_part_g, 0, sizeof(double) * b->part_g_total, st));
    BatchDev B;
    B.items = static_cast<const BItem*>(b->d_items);
    B.order = static_cast<const int32_t*>(b->d_order);
    B.passes = static_cast<const BPass*>(b->d_passes);
    B.stages = static_cast<const BStage*>(b->d_stages);
    B.ops = static_cast<const BOp*>(b->d_ops);
    B.signs = static_cast<const BSign*>(b->d_signs);
    B.czs = static_cast<const BCz*>(b->d_czs);
    B.params = static_cast<const int32_t*>(b->d_params);
    B.terms = static_cast<const BTerm*>(b->d_terms);
    B.ws = b->d_ws;
    B.energy = b->d_energy;
    B.grad = b->d_grad;
    B.part_e = b->d_part_e;
    B.part_e_off = static_cast<const int64_t*>(b->d_part_e_off);
    B.part_g = b->d_part_g;
    B.part_g_off = static_cast<const int64_t*>(b->d_part_g_off);
    B.lev_entries = static_cast<const LevelEntry*>(b->d_lev_entries);
    B.lev_pair0 = static_cast<const int32_t*>(b->d_lev_pair0);
    B.lev_pairs = static_cast<const int32_t*>(b->d_lev_pairs);
    B.lev_units = static_cast<const int32_t*>(b->d_lev_units);
    B.nlevels = nlev;
    B.counters = b->d_counter;
    B.bar_count = b->d_bar;
    B.bar_gen = b->d_bar + 1;
    B.err = b->d_err;
    B.barrier_polls = g_batch_polls.load();
    B.hold_cta = g_batch_hold.load();
    for (int c = 0; c <= kClasses; c++) B.cls_begin[c] = b->cls_begin[c];
    // cooperative launch: every CTA is resident at once, so the grid barrier cannot wait on a
    // CTA that never runs
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b->grid);
    cfg.blockDim = dim3(kBT);
    cfg.dynamicSmemBytes = b->smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    QS_TRY_CUDA(cudaLaunchKernelEx(&cfg, k_batch, B));
    QS_TRY_CUDA(cudaMemcpyAsync(b->h_err, b->d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    QS_TRY_CUDA(cudaMemcpyAsync(b->h_energy, b->d_energy, sizeof(double) * std::max(1, b->count),
                                cudaMemcpyDeviceToHost, st));
    QS_TRY_CUDA(cudaMemcpyAsync(b->h_grad, b->d_grad, sizeof(double) * std::max(1, b->total_grads),
                                cudaMemcpyDeviceToHost, st));
}

}  // namespace
}  // namespace qs

using namespace qs;

extern "C" {

#define BATCH_BEGIN \
    try {           \
        clear_error();
#define BATCH_END                                \
    }                                            \
    catch (const Error& e) {                     \
        set_error(e.msg);                        \
        return e.code;                           \
    }                                            \
    catch (const std::bad_alloc&) {              \
        set_error("host allocation failed");     \
        return QS_ERR_OOM;                       \
    }                                            \
    catch (const std::exception& e) {            \
        set_error(e.what());                     \
        return QS_ERR_CUDA;                      \
    }                                            \
    return QS_OK;

qs_status qs_batch_create(const qs_circuit* circuits, const qs_pauli_obs* observables, int count, qs_dtype dt,
                          qs_batch** out) {
    BATCH_BEGIN
    QS_REQUIRE(out != nullptr, "null output");
    *out = nullptr;
    QS_REQUIRE(count >= 1, "batch needs at least one circuit");
    QS_REQUIRE(circuits != nullptr && observables != nullptr, "null circuits or observables");
    if (dt != QS_C64) throw Error{QS_ERR_UNSUPPORTED, "batched execution runs complex64 states"};
    std::unique_ptr<qs_batch> b(new qs_batch());
    b->count = count;
    std::vector<double> cost(count);
    int param_base = 0;
    for (int k = 0; k < count; k++) {
        const qs_circuit& c = circuits[k];
        const qs_pauli_obs& o = observables[k];
        QS_REQUIRE(c.n >= 4 && c.n <= kMaxBatchQubits, "batched circuits have 4..24 qubits");
        QS_REQUIRE(c.n_gates >= 0 && (c.n_gates == 0 || c.gates), "null gate array");
        QS_REQUIRE(c.n_params >= 0, "negative parameter count");
        b->max_n = std::max(b->max_n, c.n);
        BItem it;
        std::memset(&it, 0, sizeof(it));
        it.n = c.n;
        it.angle0 = b->total_angles;
        it.grad0 = b->total_grads;
        it.ngrad = c.n_params;
        b->param0.push_back(param_base);
        std::vector<BGate> gl;
        std::vector<uint32_t> gm;
        std::vector<int32_t> gs;  // absolute angle slot of each gate (-1: none)
        int slots = 0;
        for (int i = 0; i < c.n_gates; i++) {
            const qs_gate& g = c.gates[i];
            check_qubits(c.n, g.targets, g.m, g.controls, g.mc);
            BGate bg;
            std::memset(&bg, 0, sizeof(bg));
            bg.grad = -1;
            int32_t aslot = -1;
            bg.a = uint8_t(g.targets[0]);
            uint32_t m = 1u << g.targets[0];
            QS_REQUIRE(g.kind == QS_GATE_NAMED, "batched circuits take named gates only");
            switch (g.named) {
                case QS_NAMED_RX:
                case QS_NAMED_RY:
                case QS_NAMED_RZ:
                    QS_REQUIRE(g.mc == 0 && g.m == 1, "batched rotations act on one qubit, uncontrolled");
                    bg.kind = g.named == QS_NAMED_RX ? BK_RX : g.named == QS_NAMED_RY ? BK_RY : BK_RZ;
                    aslot = b->total_angles + slots++;
                    b->angle_item.push_back(k);
                    if (g.param_index >= 0) {
                        QS_REQUIRE(g.param_index < c.n_params, "param_index out of range");
                        bg.grad = g.param_index;
                        b->angle_param.push_back(g.param_index);
                        b->angle_fixed.push_back(0.0);
                    } else {
                        b->angle_param.push_back(-1);
                        b->angle_fixed.push_back(g.params[0]);
                    }
                    break;
                case QS_NAMED_CZ:
                    QS_REQUIRE(g.m == 2 && g.mc == 0, "CZ acts on two targets");
                    bg.kind = BK_CZ;
                    bg.b = uint8_t(g.targets[1]);
                    m |= 1u << g.targets[1];
                    break;
                case QS_NAMED_CNOT:
                    QS_REQUIRE(g.m == 1 && g.mc == 1 && g.control_values[0] == 1, "CNOT has one control (value 1)");
                    bg.kind = BK_CNOT;
                    bg.b = uint8_t(g.controls[0]);
                    m |= 1u << g.controls[0];
                    break;
                case QS_NAMED_H: bg.kind = BK_H; break;
                case QS_NAMED_X: bg.kind = BK_X; break;
                case QS_NAMED_Y: bg.kind = BK_Y; break;
                case QS_NAMED_Z: bg.kind = BK_Z; break;
                default: throw Error{QS_ERR_UNSUPPORTED, "batched circuits take RX RY RZ CZ CNOT H X Y Z"};
            }
            if (g.named != QS_NAMED_CNOT) QS_REQUIRE(g.mc == 0, "only CNOT may carry a control in a batch");
            gl.push_back(bg);
            gm.push_back(m);
            gs.push_back(aslot);
        }
        b->total_angles += slots;
        b->angle_op.resize(size_t(b->total_angles));
        plan_passes(c, gl, gm, gs, *b, it);
        // observable terms
        QS_REQUIRE(o.n_terms >= 0 && (o.n_terms == 0 || (o.coef && o.x_mask && o.z_mask)), "bad observable");
        it.t0 = int(b->terms.size());
        const uint64_t lim = (1ull << c.n) - 1;
        for (int t = 0; t < o.n_terms; t++) {
            QS_REQUIRE((o.x_mask[t] & ~lim) == 0 && (o.z_mask[t] & ~lim) == 0, "Pauli term acts on a qubit >= n");
            BTerm T;
            T.xmask = uint32_t(o.x_mask[t]);
            T.zmask = uint32_t(o.z_mask[t]);
            T.coef = o.coef[t];
            T.nY = __builtin_popcount(T.xmask & T.zmask);
            T.pad = 0;
            b->terms.push_back(T);
        }
        it.t1 = int(b->terms.size());
        b->total_grads += c.n_params;
        param_base += c.n_params;
        const double passes = double(it.p1 - it.p0);
        cost[k] = std::ldexp(1.0, c.n) * (3.0 * passes + 2.0) + 64.0 * c.n_gates;
        b->items.push_back(it);
    }
    // circuits within the window: work classes by width (groups of 16, 8, 4, 2, 1 warps),
    // longest first in a class; wider circuits (class kClasses) go through the levels instead
    auto cls_of = [&](int k) {
        const int n = b->items[k].n;
        if (n > kLocal) return kClasses;
        return n == 13 ? 0 : n == 12 ? 1 : n == 11 ? 2 : n == 10 ? 3 : 4;
    };
    b->order.resize(count);
    std::iota(b->order.begin(), b->order.end(), 0);
    std::stable_sort(b->order.begin(), b->order.end(), [&](int x, int y) {
        const int cx = cls_of(x), cy = cls_of(y);
        return cx != cy ? cx < cy : cost[x] > cost[y];
    });
    for (int c = 0; c <= kClasses; c++) b->cls_begin[c] = 0;
    for (int k = 0; k < count; k++)
        if (cls_of(k) < kClasses) b->cls_begin[cls_of(k) + 1]++;
    for (int c = 0; c < kClasses; c++) b->cls_begin[c + 1] += b->cls_begin[c];
    QS_TRY_CUDA(cudaGetDevice(&b->device));
    int sms = 1;
    QS_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device));
    b->smem = 2 * sizeof(float2) * kChunk;
    QS_TRY_CUDA(cudaFuncSetAttribute(k_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, int(b->smem)));
    int per_sm = 0;
    QS_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch, kBT, b->smem));
    if (per_sm < 1) throw Error{QS_ERR_UNSUPPORTED, "batch kernel does not fit on an SM"};
    b->grid = sms * per_sm;  // all co-resident (cooperative launch)
    // circuits wider than the window get their own psi / lambda buffers and partial-sum slots,
    // and their passes become levels shared by the whole grid
    b->ws_off.assign(count, 0);
    b->part_e_off.assign(count, 0);
    b->part_g_off.assign(count, 0);
    int maxp = 0;
    std::vector<int> wide;
    for (int k = 0; k < count; k++) {
        const BItem& it = b->items[k];
        if (it.n <= kLocal) continue;
        wide.push_back(k);
        const int64_t nch = int64_t(1) << (it.n - kLocal);
        b->ws_off[k] = b->ws_amps;
        b->ws_amps += 2 * (uint64_t(1) << it.n);
        b->part_e_off[k] = b->part_e_total;
        b->part_e_total += nch;
        b->part_g_off[k] = b->part_g_total;
        b->part_g_total += nch * it.ngrad;
        maxp = std::max(maxp, it.p1 - it.p0);
    }
    // longest circuits first inside every level
    std::stable_sort(wide.begin(), wide.end(), [&](int x, int y) { return cost[x] > cost[y]; });
    auto add_level = [&](int kind, int r) {
        int units = 0;
        b->lev_pair0.push_back(kind == LV_FINAL ? ~int(b->lev_entries.size()) : int(b->lev_pairs.size()));
        for (int k : wide) {
            const BItem& it = b->items[k];
            const int np_ = it.p1 - it.p0;
            const int nch = 1 << (it.n - kLocal);
            LevelEntry e;
            e.item = k;
            e.kind = kind;
            e.unit0 = units;
            e.ws = b->ws_off[k];
            e.n = it.n;
            e.first = kind == LV_FWD && r == 0 ? 1 : 0;
            if (kind == LV_FWD) {
                if (r >= np_) continue;
                e.pass = it.p0 + r;
                units += nch;
            } else if (kind == LV_REV) {
                if (r >= np_) continue;
                e.pass = it.p1 - 1 - r;
                units += nch;
            } else if (kind == LV_LAMBDA) {
                e.pass = -1;
                units += nch;
            } else {
                e.pass = -1;
                units += 1;
            }
            if (kind != LV_FINAL)  // an even number of units: 2^(n - 13), n > 13
                b->lev_pairs.insert(b->lev_pairs.end(), size_t(units - e.unit0) / 2, int32_t(b->lev_entries.size()));
            b->lev_entries.push_back(e);
        }
        b->lev_units.push_back(units);
    };
    if (!wide.empty()) {
        for (int r = 0; r < maxp; r++) add_level(LV_FWD, r);
        add_level(LV_LAMBDA, 0);
        for (int r = 0; r < maxp; r++) add_level(LV_REV, r);
        add_level(LV_FINAL, 0);
    }
    try {
        upload(&b->d_items, b->items);
        upload(&b->d_order, b->order);
        upload(&b->d_passes, b->passes);
        upload(&b->d_stages, b->stages);
        upload(&b->d_ops, b->ops);
        upload(&b->d_signs, b->signs);
        upload(&b->d_angle_op, b->angle_op);
        upload(&b->d_czs, b->czs);
        upload(&b->d_params, b->params);
        upload(&b->d_terms, b->terms);
        QS_TRY_CUDA(dev_malloc(&b->d_theta, sizeof(double) * std::max(1, b->total_angles)));
        QS_TRY_CUDA(dev_malloc(&b->d_ws, sizeof(float2) * std::max<uint64_t>(1, b->ws_amps)));
        upload(&b->d_part_e_off, b->part_e_off);
        upload(&b->d_part_g_off, b->part_g_off);
        QS_TRY_CUDA(dev_malloc(&b->d_part_e, sizeof(double) * std::max<int64_t>(1, b->part_e_total)));
        QS_TRY_CUDA(dev_malloc(&b->d_part_g, sizeof(double) * std::max<int64_t>(1, b->part_g_total)));
        upload(&b->d_lev_entries, b->lev_entries);
        upload(&b->d_lev_pair0, b->lev_pair0);
        upload(&b->d_lev_pairs, b->lev_pairs);
        upload(&b->d_lev_units, b->lev_units);
        QS_TRY_CUDA(dev_malloc(&b->d_bar, sizeof(unsigned int) * 2));
        QS_TRY_CUDA(dev_malloc(&b->d_err, sizeof(int)));
        QS_TRY_CUDA(host_malloc_pinned(&b->h_err, sizeof(int)));
        QS_TRY_CUDA(dev_malloc(&b->d_energy, sizeof(double) * count));
        QS_TRY_CUDA(dev_malloc(&b->d_grad, sizeof(double) * std::max(1, b->total_grads)));
        QS_TRY_CUDA(dev_malloc(&b->d_counter, sizeof(unsigned int) * (kClasses + b->lev_units.size())));
        QS_TRY_CUDA(host_malloc_pinned(&b->h_theta, sizeof(double) * std::max(1, b->total_angles)));
        QS_TRY_CUDA(host_malloc_pinned(&b->h_energy, sizeof(double) * count));
        QS_TRY_CUDA(host_malloc_pinned(&b->h_grad, sizeof(double) * std::max(1, b->total_grads)));
        QS_TRY_CUDA(cudaFuncSetAttribute(k_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, int(b->smem)));
    } catch (...) {
        free_batch(b.get());
        throw;
    }
    *out = b.release();
    BATCH_END
}

qs_status qs_batch_info(const qs_batch* b, int* total_params, int* total_passes, size_t* workspace_bytes) {
    BATCH_BEGIN
    QS_REQUIRE(b != nullptr, "null batch");
    if (total_params) *total_params = b->total_grads;
    if (total_passes) *total_passes = int(b->passes.size());
    // (stages are reported through the pass count only)
    if (workspace_bytes)
        *workspace_bytes = sizeof(float2) * b->ws_amps + sizeof(double) * size_t(b->part_e_total + b->part_g_total);
    BATCH_END
}

qs_status qs_batch_traffic(const qs_batch* b, double* bytes) {
    BATCH_BEGIN
    QS_REQUIRE(b != nullptr && bytes != nullptr, "null batch or output");
    // circuits wider than the window: the first forward pass writes psi (it starts from |0..0> in
    // shared memory), every later one reads and writes it; lambda = H psi reads psi and writes
    // lambda; every reverse pass reads and writes both. Narrower circuits stay in shared memory.
    double total = 0.0;
    for (const BItem& it : b->items) {
        if (it.n <= kLocal) continue;
        const double amp = 8.0 * std::ldexp(1.0, it.n);  // complex64
        const int np_ = it.p1 - it.p0;
        if (np_ > 0) total += amp + 2.0 * amp * (np_ - 1);
        total += 2.0 * amp + 4.0 * amp * np_;
    }
    *bytes = total;
    BATCH_END
}

qs_status qs_batch_run(qs_batch* b, const double* theta, void* stream, int use_graph, double* energies,
                       double* grads) {
    BATCH_BEGIN
    QS_REQUIRE(b != nullptr && energies != nullptr, "null batch or output");
    QS_REQUIRE(b->total_grads == 0 || grads != nullptr, "null gradient output");
    // angle slots from the caller's concatenated parameters (or the gates' fixed angles)
    for (int s = 0; s < b->total_angles; s++) {
        const int p = b->angle_param[s];
        b->h_theta[s] = p >= 0 ? (theta ? theta[b->param0[b->angle_item[s]] + p] : 0.0) : b->angle_fixed[s];
    }
    QS_REQUIRE(theta != nullptr || b->total_grads == 0, "parametric batch needs theta");
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (use_graph) {
        if (b->exec && (b->graph_polls != g_batch_polls.load() || b->graph_hold != g_batch_hold.load())) {
            // the wait-test settings are kernel arguments: a graph captured under others is redone
            QS_TRY_CUDA(cudaStreamSynchronize(b->graph_stream));
            cudaGraphExecDestroy(b->exec);
            cudaGraphDestroy(b->graph);
            b->exec = nullptr;
            b->graph = nullptr;
        }
        if (!b->exec) {
            b->graph_polls = g_batch_polls.load();
            b->graph_hold = g_batch_hold.load();
            if (!b->graph_stream) QS_TRY_CUDA(cudaStreamCreateWithFlags(&b->graph_stream, cudaStreamNonBlocking));
            QS_TRY_CUDA(cudaStreamBeginCapture(b->graph_stream, cudaStreamCaptureModeThreadLocal));
            try {
                enqueue(b, b->graph_stream);
            } catch (...) {
                cudaGraph_t g = nullptr;
                cudaStreamEndCapture(b->graph_stream, &g);
                if (g) cudaGraphDestroy(g);
                throw;
            }
            QS_TRY_CUDA(cudaStreamEndCapture(b->graph_stream, &b->graph));
            QS_TRY_CUDA(cudaGraphInstantiate(&b->exec, b->graph, 0));
        }
        QS_TRY_CUDA(cudaGraphLaunch(b->exec, st));
    } else {
        enqueue(b, st);
    }
    QS_TRY_CUDA(cudaStreamSynchronize(st));
    if (*b->h_err) throw Error{QS_ERR_TIMEOUT, "batch kernel: a grid barrier wait ran out (work abandoned)"};
    std::memcpy(energies, b->h_energy, sizeof(double) * b->count);
    if (b->total_grads) std::memcpy(grads, b->h_grad, sizeof(double) * b->total_grads);
    BATCH_END
}

}  // extern "C"

namespace qs {
void batch_set_wait_polls(long long polls) { g_batch_polls.store(polls < 0 ? kBarrierSpinLimit : polls); }
void batch_set_hold_cta(bool on) { g_batch_hold.store(on ? 1 : 0); }
}  // namespace qs

extern "C" {

qs_status qs_batch_destroy(qs_batch* b) {
    BATCH_BEGIN
    if (!b) return QS_OK;
    cudaDeviceSynchronize();
    free_batch(b);
    delete b;
    BATCH_END
}

}  // extern "C"
