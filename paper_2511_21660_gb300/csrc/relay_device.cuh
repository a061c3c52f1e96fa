// Device building blocks of the fused Relay-BP kernels (paper Sec. 2.3, "Relay
// decoding"): message access, the check pass, the fault pass with decisions and
// syndrome parity, convergence and weight reductions, leg initialisation and the
// shared-memory layout.  Included by the Relay kernels and by the filtered-OSD
// kernel, whose plain-BP stage is the same passes with every gamma_j = 0.
#pragma once

#include <cuda_fp16.h>

#include "qldpc_internal.h"

namespace qldpc {
namespace {

constexpr unsigned FULL = 0xffffffffu;

template <typename MT>
struct Msg;
template <>
struct Msg<float> {
    static __device__ __forceinline__ float ld(const unsigned char *base, int off) {
        return *reinterpret_cast<const float *>(base + off);
    }
    static __device__ __forceinline__ void st(unsigned char *base, int off, float v) {
        *reinterpret_cast<float *>(base + off) = v;
    }
};
template <>
struct Msg<__half> {
    static __device__ __forceinline__ float ld(const unsigned char *base, int off) {
        return __half2float(*reinterpret_cast<const __half *>(base + off));
    }
    static __device__ __forceinline__ void st(unsigned char *base, int off, float v) {
        *reinterpret_cast<__half *>(base + off) = __float2half_rn(v);
    }
};

// Clamp to [-c, c] that keeps a NaN, as the oracle's comparisons do (fminf and fmaxf would turn it
// into -c).  Memory strengths beyond about 1e8 can overflow the two terms of lambda to opposite
// infinities; such a fault is not decided, and its messages neither bound a minimum nor turn a sign
// (a NaN from arithmetic has sign bit 0).
__device__ __forceinline__ float clampc(float x, float c) {
    float y;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(x), "f"(-c));
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(y), "f"(c));
    return y;
}

// x + h for a binary16 operand h in one float32 addition (the widening of h is exact,
// so this is __fadd_rn(x, __half2float(h)) without a separate conversion).
__device__ __forceinline__ float add_f16(float x, unsigned short h) {
    float d;
    asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(h), "f"(x));
    return d;
}

// Messages as the fault pass takes them: the stored value as it is, added to a float32 sum.
template <typename MT>
struct Raw;
template <>
struct Raw<float> {
    using T = float;
    static __device__ __forceinline__ float add(float x, float m) { return __fadd_rn(x, m); }
};
template <>
struct Raw<__half> {
    using T = unsigned short;
    static __device__ __forceinline__ float add(float x, unsigned short m) { return add_f16(x, m); }
};
template <typename MT>
__device__ __forceinline__ typename Raw<MT>::T ld_raw(const unsigned char *msg, uint32_t off) {
    return *reinterpret_cast<const typename Raw<MT>::T *>(msg + off);
}

// x + 0 = x for x != 0 and -0 + 0 = +0.  Applied to lambda(0) and to
// (1 - gamma) lambda(0) at the start of a leg, it guarantees that lambda(t) and
// therefore every stored message nu (a sum starting from lambda(t)) is never -0,
// so the check pass may read sign(nu) = -1 iff nu < 0 straight off the sign bit.
// A zero's sign never changes a comparison or a non-zero result, so this leaves
// every decision and every non-zero value as in the oracle.
__device__ __forceinline__ float canon(float x) { return __fadd_rn(x, 0.0f); }

// Weight of a decided fault in 2^-33 units, from the float's fields with integer
// operations only: |w| = m * 2^(e-23) -> m * 2^(e+10).  Exact for |w| >= 2^-10
// (smaller magnitudes are truncated); |w| < 2^20 keeps it below 2^54.
__device__ __forceinline__ long long wfix(float w) {
    const uint32_t b = __float_as_uint(w);
    const int e = (int)((b >> 23) & 0xffu) - 127;
    const long long m = (long long)((b & 0x7fffffu) | 0x800000u);
    const long long a = e >= -10 ? (m << (e + 10)) : (e > -34 ? (m >> (-10 - e)) : 0ll);
    return (b >> 31) ? -a : a;
}

// Per-fault edge list: DV byte offsets of the fault's slots (increasing check
// order); entry 0 carries the fault degree in its top byte.
template <int DV>
__device__ __forceinline__ int load_slots(const FusedGraph &g, int j, int (&sl)[DV]) {
    const int4 *p = reinterpret_cast<const int4 *>(g.var_slot + (size_t)j * DV);
    const int4 v = __ldg(p);
    sl[0] = v.x & 0xffffff;
    sl[1] = v.y;
    sl[2] = v.z;
    sl[3] = v.w;
    const int deg = (int)((unsigned)v.x >> 24);
#pragma unroll
    for (int q = 1; q < DV / 4; ++q) {
        if (deg > 4 * q) {
            const int4 u = __ldg(p + q);
            sl[4 * q] = u.x;
            sl[4 * q + 1] = u.y;
            sl[4 * q + 2] = u.z;
            sl[4 * q + 3] = u.w;
        } else {
            sl[4 * q] = sl[4 * q + 1] = sl[4 * q + 2] = sl[4 * q + 3] = 0;
        }
    }
    return deg;
}

// Swizzle of the slots inside a check (or check pair): physical position p holds
// logical slot p ^ swz(i); with 32/DC checks per 128-byte row, this spreads a
// fixed logical slot of 32 consecutive rows over 32 banks.
template <int DC>
__device__ __forceinline__ int swz(int i) {
    constexpr int sh = DC >= 32 ? 0 : (DC == 16 ? 1 : 2);
    return (i >> sh) & (DC - 1);
}

// Packed slot records of the faults of degree 2 and 3 (8 bytes a fault: x = s0 | s1 << 16,
// y = s2 | degree << 16; degree 2: s2 = s0).  Blocks of up to 3072 faults read byte offsets
// (their message arrays rarely pass 64 KB); the larger shapes read offsets in messages.
// The records are read in every fault pass: at 8 bytes the two-gross code's 64 KB stay in L1
// beside its messages, where the 16-byte table of offsets hit in half the reads.
template <typename MT, int FAULTS>
struct Packed {
    static constexpr bool kBytes = FAULTS <= kByteRecordFaults;
    static __device__ __forceinline__ const uint2 *table(const FusedGraph &g) {
        return kBytes ? g.var_rec8 : g.var_rec;
    }
    uint32_t o0, o1, o2;  // byte offsets of the fault's slots
    bool three;
    __device__ __forceinline__ explicit Packed(const uint2 q) {
        constexpr uint32_t unit = kBytes ? 1u : (uint32_t)sizeof(MT);
        o0 = (q.x & 0xffffu) * unit;
        o1 = (q.x >> 16) * unit;
        o2 = (q.y & 0xffffu) * unit;
        three = q.y >= (3u << 16);
    }
};

// Fault slots of the warp (faults threadIdx.x + r NT) that take the packed-record path: the
// slots r < n, n the number of leading slots whose 32 faults all exist and have degree 2 or 3.
// KEEP: their records stay in registers.  Set up by whole warps.
template <typename MT, int NT, int VPT, bool KEEP = false>
struct FaultSlots {
    using P = Packed<MT, NT * VPT>;
    int n;
    bool records;  // the graph has packed records
    uint2 kept[KEEP ? VPT : 1];
    __device__ __forceinline__ void init(const FusedGraph &g) {
        n = 0;
        records = P::table(g) != nullptr;
        if (!records) return;
        const int groups = (g.N + 31) >> 5;
        int r = 0;
#pragma unroll 1
        for (; r < VPT; ++r) {  // the vote makes the count uniform for the compiler
            const int q = (int)(threadIdx.x >> 5) + r * (NT / 32);
            if (!__all_sync(FULL, q < groups && __ldg(g.packed32 + q))) break;
        }
        n = r;
        if constexpr (KEEP) {
#pragma unroll
            for (int r = 0; r < VPT; ++r)
                kept[r] = r < n ? __ldg(P::table(g) + threadIdx.x + r * NT) : make_uint2(0u, 0u);
        }
    }
    __device__ __forceinline__ P get(const uint2 *rec, int r) const {  // rec: the thread's first
        if constexpr (KEEP) return P(kept[r]);
        else return P(__ldg(rec + r * NT));
    }
};

// The per-fault loops: fast(r) for the packed slots and any(r) for the others.  (One loop body
// with a branch per fault on its degree, a ballot and a bitmap store took 50 instructions a
// warp of faults, this form 31; gross code, 30,000 shots: 2.50 -> 1.96 ms with the leg
// start's same change.)  Where a warp's packed slots are all or all but the last (the detector
// models whose fault count fills their shape, as 6 to 13 rounds of the bivariate-bicycle codes do
// but for a few sizes) the loop runs without a branch between faults, which lets their loads
// overlap.  Otherwise it branches once per group of four, and takes any(r) for the whole group
// where the packed slots end (up to three packed slots a thread on the general path).
template <int VPT, typename Fast, typename Any>
__device__ __forceinline__ void each_fault(int packed, Fast fast, Any any) {
    if (packed >= VPT - 1) {
#pragma unroll
        for (int r = 0; r < VPT - 1; ++r) fast(r);
        if (packed == VPT)
            fast(VPT - 1);
        else
            any(VPT - 1);
    } else {
        constexpr int G = 4;
#pragma unroll
        for (int r0 = 0; r0 < VPT; r0 += G) {
            const int r1 = r0 + G < VPT ? r0 + G : VPT;
            if (packed >= r1) {
#pragma unroll
                for (int r = r0; r < r1; ++r) fast(r);
            } else {
#pragma unroll
                for (int r = r0; r < r1; ++r) any(r);
            }
        }
    }
}

// Start of a leg: lambda(0), Lambda(0), nu(0) and the leg's memory strengths.
//   leg 0:  lambda(0) = Lambda(0) = w
//   leg r:  Lambda(0) = previous terminal marginals; lambda(0) = Lambda(0)
//           (warm_mode 0) or w (warm_mode 1); nu(0) = lambda(0)
// bb holds (1 - gamma_j) * lambda_j(0), rounded, which is the first product of
// the memory update and is constant within a leg.
template <typename MT, int NT, int VPT, int DV, typename FS>
__device__ __forceinline__ void leg_init(const FusedGraph &g, const DevParams &p, int leg,
                                         unsigned char *msg, const FS &fs,
                                         float (&Lam)[VPT], float (&bb)[VPT],
                                         float (&gg)[VPT]) {
    const float *grow = g.gamma + (size_t)leg * g.N + threadIdx.x;
    const uint2 *rec = Packed<MT, NT * VPT>::table(g) + threadIdx.x;
    if (leg == 0 || p.warm_mode == 1) {  // lambda(0) = w
#pragma unroll
        for (int r = 0; r < VPT; ++r) {
            const int j = threadIdx.x + r * NT;
            if (j < g.N) bb[r] = canon(__ldg(g.w + j));
        }
        if (leg == 0) {
#pragma unroll
            for (int r = 0; r < VPT; ++r) Lam[r] = bb[r];
        }
    } else {  // lambda(0) = Lambda
#pragma unroll
        for (int r = 0; r < VPT; ++r) bb[r] = canon(Lam[r]);
    }
    auto fast = [&](int r) {
        const Packed<MT, NT * VPT> s = fs.get(rec, r);
        const float lam0 = bb[r], gm = __ldg(grow + r * NT);
        Msg<MT>::st(msg, s.o0, lam0);
        Msg<MT>::st(msg, s.o1, lam0);
        if (s.three) Msg<MT>::st(msg, s.o2, lam0);
        gg[r] = gm;
        bb[r] = canon(__fmul_rn(__fsub_rn(1.0f, gm), lam0));
    };
    auto any = [&](int r) {
        const int j = threadIdx.x + r * NT;
        if (j < g.N) {
            const float lam0 = bb[r], gm = __ldg(grow + r * NT);
            int sl[DV];
            const int deg = load_slots<DV>(g, j, sl);
#pragma unroll
            for (int k = 0; k < DV; ++k)
                if (k < deg) Msg<MT>::st(msg, sl[k], lam0);
            gg[r] = gm;
            bb[r] = canon(__fmul_rn(__fsub_rn(1.0f, gm), lam0));
        }
    };
    each_fault<VPT>(fs.n, fast, any);
}

// The check rule's combination of two messages: the smaller magnitude with the product of
// the signs, in one instruction (per half for a pair of binary16 values).  Exact and
// independent of the order of combination.  min, max, compare, select and logic all issue on
// the half-rate ALU pipe, which the check pass is bound by: the two smallest magnitudes, a
// select per slot and separate sign logic took 41 ALU instructions a warp of rows, this form
// 26 (gross code, 30,000 shots at p = 0.003, 384 threads: 1.96 -> 1.77 ms).
__device__ __forceinline__ float minsign(float a, float b) {
    float d;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ uint32_t minsign(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("min.xorsign.abs.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}

// o_k = the combination of rest and every a_l, l != k: pairs are combined on the way up, and
// on the way down each element meets its sibling and what lies outside the pair
// (n = 8: 20 combinations).
template <int n, typename V>
__device__ __forceinline__ void excluded(const V (&a)[n], V rest, V (&o)[n]) {
    static_assert(n >= 2 && (n & (n - 1)) == 0, "power-of-two row capacity");
    if constexpr (n == 2) {
        o[0] = minsign(a[1], rest);
        o[1] = minsign(a[0], rest);
    } else if constexpr (n == 32) {  // by groups of 8: the whole tree's values would spill
        V q[4], e[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            q[h] = a[8 * h];
#pragma unroll
            for (int k = 1; k < 8; ++k) q[h] = minsign(q[h], a[8 * h + k]);
        }
        excluded<4>(q, rest, e);
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            V x[8], y[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = a[8 * h + k];
            excluded<8>(x, e[h], y);
#pragma unroll
            for (int k = 0; k < 8; ++k) o[8 * h + k] = y[k];
        }
    } else {
        V p[n / 2], e[n / 2];
#pragma unroll
        for (int k = 0; k < n / 2; ++k) p[k] = minsign(a[2 * k], a[2 * k + 1]);
        excluded<n / 2>(p, rest, e);
#pragma unroll
        for (int k = 0; k < n / 2; ++k) {
            o[2 * k] = minsign(a[2 * k + 1], e[k]);
            o[2 * k + 1] = minsign(a[2 * k], e[k]);
        }
    }
}

// What a thread keeps for its check rows (row k of the thread: threadIdx.x + k NT; rows of
// check pairs with binary16 messages): bit k of s0 (and of s1 for the pair's second check)
// is the syndrome bit, bit k of part says that the row has padding slots.
struct RowBits {
    uint32_t s0, s1, part;
};

// Padding slots get C, which the check pass keeps there for good.
template <typename MT, int NT, int DC>
__device__ __forceinline__ void pad_rows(const FusedGraph &g, unsigned char *msg, float C) {
    const bool half = sizeof(MT) == 2;
    for (int i = threadIdx.x; i < g.Mp; i += NT) {
        const int deg = g.chk_deg[i];
        const int f = half ? swz<DC>(i >> 1) : swz<DC>(i);
        for (int k = deg; k < DC; ++k) {
            const int p = k ^ f;
            const int off = half ? (((i >> 1) * DC + p) * 4 + (i & 1) * 2) : ((i * DC + p) * 4);
            Msg<MT>::st(msg, off, C);
        }
    }
}

// The rows of the thread that have padding slots.  (Rows past the last check are never visited.)
template <typename MT, int NT, int DC>
__device__ __forceinline__ uint32_t part_rows(const FusedGraph &g) {
    uint32_t m = 0u;
    const bool half = sizeof(MT) == 2;
    const int rows = half ? (g.M + 1) >> 1 : g.M;
    for (int i = threadIdx.x, k = 0; i < rows; i += NT, ++k) {
        const bool full = half ? g.chk_deg[2 * i] == DC && g.chk_deg[2 * i + 1] == DC
                               : g.chk_deg[i] == DC;
        m |= (full ? 0u : 1u) << k;
    }
    return m;
}

template <typename MT, int NT, int DC>
__device__ __forceinline__ uint32_t setup_rows(const FusedGraph &g, unsigned char *msg, float C) {
    pad_rows<MT, NT, DC>(g, msg, C);
    return part_rows<MT, NT, DC>(g);
}

// The syndrome bits of the thread's rows, from the shot's packed words in global memory.
template <typename MT, int NT>
__device__ __forceinline__ void row_syndromes(const FusedGraph &g, const uint64_t *sy,
                                              RowBits &rb) {
    rb.s0 = rb.s1 = 0u;
    const uint32_t *w = reinterpret_cast<const uint32_t *>(sy);
    const bool half = sizeof(MT) == 2;
    const int rows = half ? (g.M + 1) >> 1 : g.M;
#pragma unroll 1
    for (int i = threadIdx.x, k = 0; i < rows; i += NT, ++k) {
        if (half) {
            const uint32_t b = __ldg(w + (i >> 4)) >> (2 * (i & 15));
            rb.s0 |= (b & 1u) << k;
            rb.s1 |= ((b >> 1) & 1u) << k;
        } else {
            rb.s0 |= ((__ldg(w + (i >> 5)) >> (i & 31)) & 1u) << k;
        }
    }
}

// The parity words start an iteration as the syndrome.
template <int NT>
__device__ __forceinline__ void set_parity(const FusedGraph &g, const uint32_t *sg,
                                           uint32_t *par) {
    if (threadIdx.x >= g.m_words) return;
    par[threadIdx.x] = sg[threadIdx.x];
    for (int q = threadIdx.x + NT; q < g.m_words; q += NT) par[q] = sg[q];
}

// Check pass, float32 messages: mu_{i->j}(t) from nu(t-1) for every check, in place.
// Slot k gets the combination of every other slot of the row and of (-1)^sigma_i C: the
// smallest other magnitude, at most C, with the product of the other signs and the check's.
// The minimum with C also stands for the clamp of nu to [-C, C]: min(|nu|, C) is the clamped
// magnitude and a clamp keeps the sign, so the fault pass stores nu unclamped.
// Padding slots hold +C, the neutral value here, and keep it.
// Slots are processed in physical order: the rule does not depend on the order.
// Lanes read and write their row's 16-byte chunks in the order k4 ^ cs: rows are
// 4*DC bytes apart, and cs = (row / rows per 128-byte line) mod chunks per row makes
// each 128-bit access of a warp touch every bank equally often (no bank conflict).
// NT is a multiple of 32, so cs and the swizzle are the same for all rows of a thread.
// The parity words start the iteration as the syndrome (the fault pass flips them to 0).
template <int NT, int DC>
__device__ __forceinline__ void check_pass(const FusedGraph &g, float *msg, const uint32_t *sg,
                                           uint32_t *par, const RowBits &rb, float C) {
    set_parity<NT>(g, sg, par);
    static_assert(NT % 32 == 0, "the chunk order and the swizzle repeat every 32 rows");
    const int cs = (threadIdx.x / (DC >= 32 ? 1 : 32 / DC)) & (DC / 4 - 1);  // chunk order
    const uint32_t c = __float_as_uint(C);
    float4 *row = reinterpret_cast<float4 *>(msg + (size_t)threadIdx.x * DC);
    uint32_t sb = rb.s0, part = rb.part;
#pragma unroll 1
    for (int i = threadIdx.x; i < g.M; i += NT) {
        float v[DC], o[DC];
#pragma unroll
        for (int k4 = 0; k4 < DC / 4; ++k4) {
            const float4 t = row[k4 ^ cs];
            v[4 * k4] = t.x;
            v[4 * k4 + 1] = t.y;
            v[4 * k4 + 2] = t.z;
            v[4 * k4 + 3] = t.w;
        }
        excluded<DC>(v, __uint_as_float((sb << 31) | c), o);
#pragma unroll
        for (int k4 = 0; k4 < DC / 4; ++k4)
            row[k4 ^ cs] = make_float4(o[4 * k4], o[4 * k4 + 1], o[4 * k4 + 2], o[4 * k4 + 3]);
        if (part & 1u) {  // padding slots get C back: the last slot, seldom more
            float *r = reinterpret_cast<float *>(row);
            r[(DC - 1) ^ swz<DC>(threadIdx.x)] = C;
            if (g.min_deg < DC - 1)
                for (int k = g.chk_deg[i]; k < DC - 1; ++k) r[k ^ swz<DC>(threadIdx.x)] = C;
        }
        row += NT * DC / 4;
        sb >>= 1;
        part >>= 1;
    }
}

// Check pass, binary16 messages: checks 2q and 2q+1 share each 32-bit word (low
// and high half), processed together; minima and signs are exact in any format.  A per-pair
// mask keeps C in padding halves.
// Row chunks are visited in the order k4 ^ cs as in the float32 pass (rows of check
// pairs are 4*DC bytes apart too); only the padding mask follows the order.
template <int NT, int DC>
__device__ __forceinline__ void check_pass(const FusedGraph &g, __half *msg, const uint32_t *sg,
                                           uint32_t *par, const RowBits &rb, float C) {
    set_parity<NT>(g, sg, par);
    const __half2 C2 = __float2half2_rn(C);
    const uint32_t c2 = *reinterpret_cast<const uint32_t *>(&C2);
    const int M2 = (g.M + 1) >> 1;
    const int cs = (threadIdx.x / (DC >= 32 ? 1 : 32 / DC)) & (DC / 4 - 1);
    uint4 *row = reinterpret_cast<uint4 *>(msg + (size_t)threadIdx.x * 2 * DC);
    uint32_t sb0 = rb.s0, sb1 = rb.s1, part = rb.part;
#pragma unroll 1
    for (int q = threadIdx.x; q < M2; q += NT) {
        const uint32_t sx = (sb1 << 31) | ((sb0 & 1u) << 15);
        uint32_t v[DC];
#pragma unroll
        for (int k4 = 0; k4 < DC / 4; ++k4) {
            const uint4 t = row[k4 ^ cs];
            v[4 * k4] = t.x;
            v[4 * k4 + 1] = t.y;
            v[4 * k4 + 2] = t.z;
            v[4 * k4 + 3] = t.w;
        }
        uint32_t o[DC];
        excluded<DC>(v, c2 | sx, o);
        if (part & 1u) {
            const uint4 *pm4 = reinterpret_cast<const uint4 *>(g.pad_mask + (size_t)q * DC);
#pragma unroll
            for (int k4 = 0; k4 < DC / 4; ++k4) {
                const uint4 t = __ldg(pm4 + (k4 ^ cs));
                o[4 * k4] = (o[4 * k4] & ~t.x) | (c2 & t.x);
                o[4 * k4 + 1] = (o[4 * k4 + 1] & ~t.y) | (c2 & t.y);
                o[4 * k4 + 2] = (o[4 * k4 + 2] & ~t.z) | (c2 & t.z);
                o[4 * k4 + 3] = (o[4 * k4 + 3] & ~t.w) | (c2 & t.w);
            }
        }
#pragma unroll
        for (int k4 = 0; k4 < DC / 4; ++k4)
            row[k4 ^ cs] = make_uint4(o[4 * k4], o[4 * k4 + 1], o[4 * k4 + 2], o[4 * k4 + 3]);
        row += NT * DC / 4;
        sb0 >>= 1;
        sb1 >>= 1;
        part >>= 1;
    }
}

// Fault update for one fault: marginal and excluded sums (increasing check order, one
// rounding per addition, as written in the oracle).  A slot the fault does not have adds
// +0, which changes no sum (none is -0: they start from lambda, which canon keeps from
// -0).  Messages are stored unclamped (the check pass takes their magnitudes' minimum
// with C); the marginal is clamped.
//
// Faults of degree 2 and 3, by the byte offsets of their slots.
template <typename MT>
__device__ __forceinline__ float fault_update(unsigned char *msg, uint32_t o0, uint32_t o1,
                                              uint32_t o2, bool three, float lam, float C) {
    using R = Raw<MT>;
    const typename R::T m0 = ld_raw<MT>(msg, o0), m1 = ld_raw<MT>(msg, o1);
    typename R::T m2 = 0;
    if (three) m2 = ld_raw<MT>(msg, o2);
    const float p1 = R::add(lam, m0), p2 = R::add(p1, m1);
    Msg<MT>::st(msg, o0, R::add(R::add(lam, m1), m2));
    Msg<MT>::st(msg, o1, R::add(p1, m2));
    if (three) Msg<MT>::st(msg, o2, p2);
    const float L = R::add(p2, m2);
    return clampc(L, C);
}
template <typename MT, int FAULTS>
__device__ __forceinline__ float fault_update(unsigned char *msg, const Packed<MT, FAULTS> &s,
                                              float lam, float C) {
    return fault_update<MT>(msg, s.o0, s.o1, s.o2, s.three, lam, C);
}

// Any degree up to DV.  Where that is 8, degrees 2 and 3 of a graph without packed records (more
// than 64 KB of messages, up to 3072 faults) have their own code here too: the loop below takes 36
// additions whatever the degree (16-slot rows, 1500 checks, 2400 faults of degree 3, 6000 shots:
// 0.70 -> 0.64 ms; 32-slot rows, 600 checks, 2900 faults: 10.6 -> 9.2).  With records, what comes
// here are warps of mixed degrees, which the branch would only split (16-slot rows, degrees 3 to
// 5: 0.60 -> 0.64 ms; 8-slot rows, degrees 3 and 4: 0.26 -> 0.31).
// CUT: values above C are cut to it before the store.  The check pass bounds them anyway; the decode
// kernels of the 8-slot float32 family do it because without this instruction the compiler spills 8
// bytes in the iteration loop of the 256 x 11 shape (10^5 gross shots 4.68 -> 4.74 ms).
template <typename MT, int DV, bool CUT = false>
__device__ __forceinline__ float fault_update(unsigned char *msg, const int (&sl)[DV], int deg,
                                              bool records, float lam, float C) {
    using R = Raw<MT>;
    if (DV > 4 && !records && (deg == 2 || deg == 3))
        return fault_update<MT>(msg, sl[0], sl[1], sl[2], deg == 3, lam, C);
    typename R::T mu[DV];
#pragma unroll
    for (int k = 0; k < DV; ++k) {
        mu[k] = 0;
        if (k < deg) mu[k] = ld_raw<MT>(msg, sl[k]);
    }
    float p = lam;  // lam + mu_0 + .. + mu_{k-1}
#pragma unroll
    for (int k = 0; k < DV; ++k) {
        float v = p;
#pragma unroll
        for (int k2 = k + 1; k2 < DV; ++k2) v = R::add(v, mu[k2]);
        if (CUT) asm("min.NaN.f32 %0, %1, %2;" : "=f"(v) : "f"(v), "f"(C));
        if (k < deg) Msg<MT>::st(msg, sl[k], v);
        p = R::add(p, mu[k]);
    }
    return clampc(p, C);
}

// Check of a message slot from its byte offset.
template <typename MT, int DC>
__device__ __forceinline__ int check_of_slot(int off) {
    if (sizeof(MT) == 2) return 2 * (off / (4 * DC)) + ((off >> 1) & 1);
    return off / (4 * DC);
}

// Fault pass: memory update, marginals, fault->check messages, decisions into the
// bitmap fw, and the syndrome of the decision: every fault with F_j = 1 flips the
// parity bits of its checks in par (the preceding check pass set it to the syndrome, so
// all words end 0 iff H F = sigma).  Decisions are sparse, so this costs a few atomics
// per shot instead of a pass over all edges.
// The decision of a fault is the sign bit of its marginal (never -0, see fault_update), shifted
// into a mask; the bitmap words and the parity flips follow for the warps that decided any.
// Returns the thread's decided faults (bit VPT-1-r: fault threadIdx.x + r*NT has F_j = 1).
template <typename MT, int NT, int VPT, int DC, int DV, bool CUT = false, typename FS>
__device__ __forceinline__ uint32_t fault_pass(const FusedGraph &g, unsigned char *msg, uint32_t *fw,
                                           uint32_t *par, const FS &fs, float (&Lam)[VPT],
                                           const float (&bb)[VPT], const float (&gg)[VPT],
                                           float C) {
    static_assert(VPT <= 32, "one decision bit per fault of the thread");
    const int lane = threadIdx.x & 31, wb = threadIdx.x & ~31;
    const uint2 *rec = Packed<MT, NT * VPT>::table(g) + threadIdx.x;
    uint32_t dmask = 0u;
    auto decide = [&](float L) {
        dmask = __funnelshift_l(__float_as_uint(L), dmask, 1);  // dmask << 1 | sign(L)
    };
    auto fast = [&](int r) {
        const Packed<MT, NT * VPT> s = fs.get(rec, r);
        const float lam = __fadd_rn(bb[r], __fmul_rn(gg[r], Lam[r]));
        Lam[r] = fault_update(msg, s, lam, C);
        decide(Lam[r]);
    };
    auto any = [&](int r) {
        const int j = threadIdx.x + r * NT;
        float L = 0.0f;
        if (j < g.N) {
            const float lam = __fadd_rn(bb[r], __fmul_rn(gg[r], Lam[r]));
            int sl[DV];
            const int deg = load_slots<DV>(g, j, sl);
            L = fault_update<MT, DV, CUT>(msg, sl, deg, fs.records, lam, C);
            Lam[r] = L;
        }
        decide(L);
    };
    each_fault<VPT>(fs.n, fast, any);
    __syncwarp();
    // bitmap words of the warp: fault slot r's 32 faults are word (wb + r NT) / 32
    uint32_t word = 0u;
    if (__any_sync(FULL, dmask != 0u)) {
#pragma unroll
        for (int r = 0; r < VPT; ++r) {
            const uint32_t bal = __ballot_sync(FULL, (dmask >> (VPT - 1 - r)) & 1u);
            if (lane == r) word = bal;
        }
        // decided faults are few: flip their checks' parity
        for (uint32_t m = dmask; m; m &= m - 1u) {
            const int r = VPT - __ffs(m);
            int sl[DV];
            const int deg = load_slots<DV>(g, threadIdx.x + r * NT, sl);
#pragma unroll
            for (int k = 0; k < DV; ++k)
                if (k < deg) {
                    const int c = check_of_slot<MT, DC>(sl[k]);
                    atomicXor(par + (c >> 5), 1u << (c & 31));
                }
        }
    }
    if (lane < VPT && wb + lane * NT < g.N) fw[(wb + lane * NT) >> 5] = word;
    return dmask;
}

// H F = sigma ?  (every parity word 0)  Each warp looks on its own (no block barrier);
// every warp reaches the same answer.
__device__ __forceinline__ bool warp_converged(const uint32_t *par, int nw) {
    const int lane = threadIdx.x & 31;
    uint32_t bad = lane < nw ? par[lane] : 0u;
    for (int q = lane + 32; q < nw; q += 32) bad |= par[q];
    return !__any_sync(FULL, bad != 0u);
}

// Adds this thread's share of the solution weight sum_j F_j w_j (2^-33 units) to the
// block's accumulator: only the few threads with decided faults (mask dm from the
// fault pass, bit VPT-1-r for fault r) issue an atomic.  Integer addition makes the total exact and
// independent of the order.
template <int NT, int VPT>
__device__ __forceinline__ void add_weight(const FusedGraph &g, uint32_t dm, long long *acc) {
    long long w = 0;
    for (uint32_t m = dm; m; m &= m - 1u) w += wfix(__ldg(g.w + threadIdx.x + (VPT - __ffs(m)) * NT));
    if (w != 0)
        atomicAdd(reinterpret_cast<unsigned long long *>(acc), (unsigned long long)w);
}

template <int NT>
__device__ __forceinline__ void store_bits(uint64_t *dst, const uint32_t *fw, int words) {
    for (int q = threadIdx.x; q < words; q += NT)
        dst[q] = (uint64_t)fw[2 * q] | ((uint64_t)fw[2 * q + 1] << 32);
}

// Kept solution: the output row and the shared copy used by warp_same_solution.
template <int NT>
__device__ __forceinline__ void keep_solution(uint64_t *dst, const uint32_t *fw, uint32_t *fb,
                                              int words) {
    for (int q = threadIdx.x; q < words; q += NT) {
        const uint32_t lo = fw[2 * q], hi = fw[2 * q + 1];
        fb[2 * q] = lo;
        fb[2 * q + 1] = hi;
        dst[q] = (uint64_t)lo | ((uint64_t)hi << 32);
    }
}

// Shared memory: messages [msg_bytes], decision bitmap fw [f_words], kept solution
// fb [f_words], syndrome sg [2*syn_words] (bits past M cleared), two parity buffers
// par [2][m_words].  (The prior LLRs are read from global memory, once a shot and for the
// decided faults of a solution.)
__device__ __forceinline__ void smem_layout(const FusedGraph &g, unsigned char *raw,
                                            uint32_t *&fw, uint32_t *&fb, uint32_t *&sg,
                                            uint32_t *&par) {
    const size_t mb = ((size_t)g.msg_bytes + 15) & ~(size_t)15;
    fw = reinterpret_cast<uint32_t *>(raw + mb);
    fb = fw + g.f_words;
    sg = fb + g.f_words;
    par = sg + 2 * g.syn_words;
}

// Plain min-sum BP (paper Sec. 2.3, "Belief propagation decoding"): DMem-BP with every
// gamma_j = 0, which the graph's gamma row (all zeros) provides, from the priors, for
// `iters` iterations without early exit; the marginals end in Lam.  Re-stages the
// padding slots first (callers reuse the message area between shots).
// Called by every thread of the block.
template <int NT, int VPT, int DC, int DV>
__device__ __forceinline__ void plain_bp(const FusedGraph &g, const DevParams &p, int iters,
                                         const uint64_t *sy, unsigned char *msg, uint32_t *fw,
                                         uint32_t *sg, uint32_t *par,
                                         float (&Lam)[VPT], float (&bb)[VPT], float (&gg)[VPT]);

// Is the decision bitmap equal to the kept solution (its first `words` words)?  Each
// warp decides on its own, comparing 128 bits per lane: fw and fb are 16-byte aligned,
// f_words is a multiple of 4 and the words past the last fault are zero in both.
__device__ __forceinline__ bool warp_same_solution(const uint32_t *fw, const uint32_t *fb,
                                                   int words) {
    const uint4 *a = reinterpret_cast<const uint4 *>(fw), *b = reinterpret_cast<const uint4 *>(fb);
    uint32_t diff = 0;
    for (int q = threadIdx.x & 31; 4 * q < words; q += 32) {
        const uint4 x = a[q], y = b[q];
        diff |= (x.x ^ y.x) | (x.y ^ y.y) | (x.z ^ y.z) | (x.w ^ y.w);
    }
    return !__any_sync(FULL, diff != 0u);
}

// Once a block: the bitmaps' words past the last fault stay zero.
template <int NT>
__device__ __forceinline__ void clear_bitmaps(const FusedGraph &g, uint32_t *fw) {
    for (int q = threadIdx.x; q < 2 * g.f_words; q += NT) fw[q] = 0u;  // fw and fb
}

template <int NT>
__device__ __forceinline__ void load_syndrome(const FusedGraph &g, const uint64_t *sy,
                                              uint32_t *sg) {
    for (int q = threadIdx.x; q < g.syn_words; q += NT) {
        uint64_t v = __ldg(sy + q);
        const int hi = g.M - 64 * q;  // padding bits of the last word are ignored
        if (hi < 64) v &= (1ull << hi) - 1ull;
        sg[2 * q] = (uint32_t)v;
        sg[2 * q + 1] = (uint32_t)(v >> 32);
    }
}


template <int NT, int VPT, int DC, int DV>
__device__ __forceinline__ void plain_bp(const FusedGraph &g, const DevParams &p, int iters,
                                         const uint64_t *sy, unsigned char *msg, uint32_t *fw,
                                         uint32_t *sg, uint32_t *par,
                                         float (&Lam)[VPT], float (&bb)[VPT], float (&gg)[VPT]) {
    clear_bitmaps<NT>(g, fw);
    load_syndrome<NT>(g, sy, sg);
    FaultSlots<float, NT, VPT> fs;
    fs.init(g);
    RowBits rb;
    rb.part = setup_rows<float, NT, DC>(g, msg, p.clip);
    row_syndromes<float, NT>(g, sy, rb);
    __syncthreads();
    leg_init<float, NT, VPT, DV>(g, p, 0, msg, fs, Lam, bb, gg);
    __syncthreads();
    for (int t = 0; t < iters; ++t) {
        check_pass<NT, DC>(g, reinterpret_cast<float *>(msg), sg, par, rb, p.clip);
        __syncthreads();
        fault_pass<float, NT, VPT, DC, DV>(g, msg, fw, par, fs, Lam, bb, gg, p.clip);
        __syncthreads();
    }
}

}  // namespace
}  // namespace qldpc
