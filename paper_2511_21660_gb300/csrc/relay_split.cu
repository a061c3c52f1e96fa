// Resuming launch of the tail continuation with one shot spread over a cluster of blocks.
//
// The shots that reach this launch run thousands of iterations and there are few of them, so
// what counts is the time of one iteration of one shot.  On one SM that is bound by the SM's
// own issue and shared-memory rate (gross code, 1024 threads: 1.68 us; here 1.2-1.3).  Here each block of a
// cluster of kSplit holds a contiguous range of checks with their message rows in its shared
// memory, and the faults whose first check lies there.  The check pass is local; the fault
// pass reads and writes the few rows of other blocks through distributed shared memory (in a
// detector model that is the measurement faults between the ranges); the passes are separated
// by cluster barriers.  Every block keeps the leg schedule of the shot and reaches the same
// decisions.  The arithmetic and its order are the decode kernels', so results are
// bit-identical to theirs.
//
// What an iteration takes is latency: two cluster barriers with release and acquire (360
// cycles each, 500 behind remote stores), remote reads (217), the passes.  So the convergence
// test adds no step of its own: the fault pass stores each fault's decision, a byte per
// message, beside its messages, and the threads of the next check pass fold their rows' bytes
// into one flag a block, which every block reads with its next messages.  That check pass is
// then one too many when the leg has ended, which costs nothing: the next leg's start
// overwrites every message.  (Parity words flipped by atomics and read by all blocks after the
// second barrier took 1.55 us an iteration instead of 1.3.)
#include "relay_device.cuh"
#include "relay_split.h"

namespace qldpc {
namespace {

constexpr int DC = 8, DV = 4;  // the family of rows up to 8 slots and faults up to 4

__device__ __forceinline__ uint32_t shared_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
// The address of block `rank`'s copy of a shared location; one's own keeps its address.
__device__ __forceinline__ uint32_t peer_addr(uint32_t own, int rank, int me) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(own), "r"(rank));
    return rank == me ? own : a;
}
__device__ __forceinline__ uint32_t peer_ld(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ long long peer_ld64(uint32_t a) {
    long long v;
    asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void peer_st8(uint32_t a, uint32_t v) {
    asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
template <typename MT>
struct Peer;
template <>
struct Peer<float> {
    static __device__ __forceinline__ float ld(uint32_t a) { return __uint_as_float(peer_ld(a)); }
    static __device__ __forceinline__ void st(uint32_t a, float v) {
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
    }
};
template <>
struct Peer<__half> {
    static __device__ __forceinline__ unsigned short ld(uint32_t a) {
        unsigned short v;
        asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
        return v;
    }
    static __device__ __forceinline__ void st(uint32_t a, float v) {
        const unsigned short h = __half_as_ushort(__float2half_rn(v));
        asm volatile("st.shared::cluster.u16 [%0], %1;" ::"r"(a), "h"(h) : "memory");
    }
};

// Decision bytes lie in the order of the messages: 8 to a row, and with binary16 messages 16 to
// a pair of rows, whose bytes alternate.
template <typename MT>
__device__ __forceinline__ uint32_t decision_byte(uint32_t msg_off) {
    return msg_off / (uint32_t)sizeof(MT);
}

// Parity of the decisions of row i.
template <typename MT>
__device__ __forceinline__ uint32_t row_parity(const unsigned char *dec, int i) {
    if (sizeof(MT) == 4) {
        const uint2 x = reinterpret_cast<const uint2 *>(dec)[i];
        return __popc(x.x ^ x.y) & 1u;
    }
    const uint4 x = reinterpret_cast<const uint4 *>(dec)[i >> 1];
    const uint32_t half = (i & 1) ? 0xff00ff00u : 0x00ff00ffu;
    return __popc((x.x ^ x.y ^ x.z ^ x.w) & half) & 1u;
}

template <typename MT, int NT, int VPT, int DVU, int MINB>
__global__ void __cluster_dims__(kSplit, 1, 1) __launch_bounds__(NT, MINB)
    split_resume(SplitGraph g, DevParams p, const uint64_t *__restrict__ syn, DecodeOut out,
                 unsigned int *counter, ShotMap map, TailCont tc, int most) {
    using R = Raw<MT>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *msg = smem_raw;
    unsigned char *dec = smem_raw + g.msg_bytes;  // decision of each message's fault, a byte
    __shared__ uint32_t s_zero, s_trash;  // read and written for the slots a fault does not have
    __shared__ int s_take;
    __shared__ uint32_t s_bad[2], s_diff;
    __shared__ long long s_w[2];
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int tid = threadIdx.x, lane = tid & 31;
    const int me = (int)(blockIdx.x % kSplit), cluster = (int)(blockIdx.x / kSplit);
    const int n = (int)min(*tc.count, (unsigned int)tc.cap);
    // the whole cluster, as are all of them when one block a shot is faster (see
    // launch_persistent)
    if (cluster >= n || n > most) return;

    // this block's rows as a graph of their own, for the check pass
    const int row0 = g.row0[me];
    FusedGraph lg{};
    lg.M = g.row0[me + 1] - row0;
    lg.Mp = lg.M + (lg.M & 1);
    lg.m_words = 0;  // the check pass sets no parity words
    lg.min_deg = g.min_deg;
    lg.chk_deg = g.chk_deg + row0;
    lg.pad_mask = g.pad_mask + (size_t)me * g.pad_stride;
    const float C = p.clip;
    RowBits rb;
    rb.part = setup_rows<MT, NT, DC>(lg, msg, C);

    // this thread's faults and the addresses of their messages
    int fj[VPT];
    uint32_t at[VPT][DVU], bit[VPT][DVU];  // addresses of the messages and decision bytes
    const uint32_t zero = shared_addr(&s_zero), trash = shared_addr(&s_trash);
#pragma unroll
    for (int v = 0; v < VPT; ++v) {
        const size_t q = (size_t)me * (NT * VPT) + tid + v * NT;
        fj[v] = g.fault[q];
        const uint4 s = g.slots[q];
        const uint32_t e[DV] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int k = 0; k < DVU; ++k) {
            const uint32_t off = e[k] & 0xffffffu;
            const int b = (int)(e[k] >> 24);
            at[v][k] = e[k] == kNoSlot ? zero : peer_addr(shared_addr(msg) + off, b, me);
            bit[v][k] = e[k] == kNoSlot
                            ? trash
                            : peer_addr(shared_addr(dec) + decision_byte<MT>(off), b, me);
        }
    }
    for (int q = tid; q < g.rows * DC / 4; q += NT) reinterpret_cast<uint32_t *>(dec)[q] = 0u;
    const uint32_t flag = peer_addr(shared_addr(s_bad), lane < kSplit ? lane : me, me);
    if (tid == 0) s_zero = s_bad[0] = s_bad[1] = 0u;
    if (tid == 0) s_w[0] = s_w[1] = 0;
    int ab = 0;

    for (;;) {
        cluster_sync();  // every block is done with the previous shot
        if (me == 0 && tid == 0) s_take = (int)atomicAdd(counter, 1u);
        cluster_sync();
        const int rec = (int)peer_ld(peer_addr(shared_addr(&s_take), 0, me));
        if (rec >= n) break;  // every block of the cluster
        const TailRecord r = tc.rec[rec];
        int leg = r.leg, sols = r.sols;
        long long iters = r.iters, best = r.Wbest;
        const uint64_t *sy = syn + (size_t)r.shot * map.syn_stride;
        uint32_t *cor = reinterpret_cast<uint32_t *>(out.corr + (size_t)r.shot * map.cor_stride);
        // the rows' syndrome: bits by row, and words from bit row0 on
        const uint32_t *sw = reinterpret_cast<const uint32_t *>(sy);
        rb.s0 = rb.s1 = 0u;
        const int rows = sizeof(MT) == 2 ? (lg.M + 1) >> 1 : lg.M;
        for (int i = tid, k = 0; i < rows; i += NT, ++k) {
            const int b = row0 + (sizeof(MT) == 2 ? 2 * i : i);
            const uint32_t x = __ldg(sw + (b >> 5)) >> (b & 31);  // row0 is even
            rb.s0 |= (x & 1u) << k;
            rb.s1 |= ((x >> 1) & 1u) << k;
        }
        uint32_t odd = 0u;  // bit k: syndrome bit of row tid + k NT
        for (int i = tid, k = 0; i < lg.M; i += NT, ++k)
            odd |= ((__ldg(sw + ((row0 + i) >> 5)) >> ((row0 + i) & 31)) & 1u) << k;
        float Lam[VPT], bb[VPT], gg[VPT];
        uint32_t kept = 0u, dm = 0u;  // bit v: fault v in the kept solution, decided now
#pragma unroll
        for (int v = 0; v < VPT; ++v) {
            Lam[v] = bb[v] = gg[v] = 0.0f;
            if (fj[v] < 0) continue;
            Lam[v] = tc.lam[(size_t)rec * g.N + fj[v]];
            if (sols > 0) kept |= ((cor[fj[v] >> 5] >> (fj[v] & 31)) & 1u) << v;
        }
        int turn = 0;  // copy of s_bad in use
        for (;;) {  // legs
            const float *grow = g.gamma + (size_t)leg * g.N;
#pragma unroll
            for (int v = 0; v < VPT; ++v) {
                if (fj[v] < 0) continue;
                const float lam0 =
                    canon(leg == 0 || p.warm_mode == 1 ? __ldg(g.w + fj[v]) : Lam[v]);
                if (leg == 0) Lam[v] = lam0;
                const float gm = __ldg(grow + fj[v]);
                gg[v] = gm;
                bb[v] = canon(__fmul_rn(__fsub_rn(1.0f, gm), lam0));
#pragma unroll
                for (int k = 0; k < DVU; ++k) Peer<MT>::st(at[v][k] == zero ? trash : at[v][k], lam0);
            }
            cluster_sync();  // the leg's initial messages
            int limit = leg == 0 ? p.T1 : p.T2;
            if (p.max_iters > 0) {
                const long long left = p.max_iters - iters;
                limit = left < limit ? (left < 1 ? 1 : (int)left) : limit;
            }
            bool conv = false;
            for (int t = 0;; ++t) {
                // check pass, and whether iteration t's decisions leave a row unsatisfied
                check_pass<NT, DC>(lg, reinterpret_cast<MT *>(msg), nullptr, nullptr, rb, C);
                bool bad = false;
                for (int i = tid, k = 0; i < lg.M; i += NT, ++k) {
                    bad |= row_parity<MT>(dec, i) != ((odd >> k) & 1u);
                }
                if (__any_sync(FULL, bad) && lane == 0) s_bad[turn] = 1u;
                cluster_sync();
                const uint32_t seen = peer_ld(flag + 4u * (uint32_t)turn);
                typename R::T mu[VPT][DVU];  // all reads first: remote ones take longest
#pragma unroll
                for (int v = 0; v < VPT; ++v)
#pragma unroll
                    for (int k = 0; k < DVU; ++k) mu[v][k] = Peer<MT>::ld(at[v][k]);
                turn ^= 1;
                if (tid == 0) s_bad[turn] = 0u;
                conv = t > 0 && !__any_sync(FULL, seen != 0u);
                if (conv || t == limit) {
                    iters += t;
                    break;
                }
                dm = 0u;
#pragma unroll
                for (int v = 0; v < VPT; ++v) {
                    const float lam = __fadd_rn(bb[v], __fmul_rn(gg[v], Lam[v]));
                    float s = lam;  // lam + mu_0 + .. + mu_{k-1}
#pragma unroll
                    for (int k = 0; k < DVU; ++k) {
                        float x = s;
#pragma unroll
                        for (int k2 = k + 1; k2 < DVU; ++k2) x = R::add(x, mu[v][k2]);
                        Peer<MT>::st(at[v][k] == zero ? trash : at[v][k], x);
                        s = R::add(s, mu[v][k]);
                    }
                    Lam[v] = clampc(s, C);
                    const uint32_t d = __float_as_uint(Lam[v]) >> 31;
                    dm |= d << v;
#pragma unroll
                    for (int k = 0; k < DVU; ++k) peer_st8(bit[v][k], d);
                }
                cluster_sync();
            }
            cluster_sync();  // s_bad and the messages have been read
            if (conv) {  // the solution's weight and whether it is the kept one, over the cluster
                long long w = 0;
#pragma unroll
                for (int v = 0; v < VPT; ++v)
                    if ((dm >> v) & 1u) w += wfix(__ldg(g.w + fj[v]));
                if (w != 0)
                    atomicAdd(reinterpret_cast<unsigned long long *>(s_w + ab),
                              (unsigned long long)w);
                const int diff = __syncthreads_or(dm != kept);
                if (tid == 0) s_diff = diff ? 1u : 0u;
                cluster_sync();
                long long W = 0;
                uint32_t differs = 0u;
                for (int b = 0; b < kSplit; ++b) {
                    W += peer_ld64(peer_addr(shared_addr(s_w + ab), b, me));
                    differs |= peer_ld(peer_addr(shared_addr(&s_diff), b, me));
                }
                if (tid == 0) s_w[ab ^ 1] = 0;
                ab ^= 1;
                if (sols == 0 || (differs && W < best)) {
                    kept = dm;
                    best = W;
                }
                ++sols;
                cluster_sync();  // s_w and s_diff have been read
            }
            const bool done = sols >= p.S || leg == p.R || (p.max_iters > 0 && iters >= p.max_iters);
            ++leg;
            if (done) break;
        }
        // the correction: the kept solution, or the last decision when there is none
        const uint32_t bits = sols > 0 ? kept : dm;
        if (me == 0)
            for (int q = tid; q < 2 * g.cor_words; q += NT) cor[q] = 0u;
        cluster_sync();
#pragma unroll
        for (int v = 0; v < VPT; ++v)
            if ((bits >> v) & 1u) atomicOr(cor + (fj[v] >> 5), 1u << (fj[v] & 31));
        if (me == 0 && tid == 0) {
            if (out.legs) out.legs[r.shot] = leg;
            if (out.conv) out.conv[r.shot] = sols > 0 ? 1 : 0;
            if (out.iters) out.iters[r.shot] = (int32_t)iters;
        }
    }
    cluster_sync();  // no block leaves while another may read its shared memory
}

template <typename MT, int NT, int VPT, int DVU, int MINB>
cudaError_t launch_split(int clusters, size_t smem, cudaStream_t st, const SplitGraph &g,
                         const DevParams &p, const uint64_t *syn, DecodeOut out,
                         unsigned int *counter, ShotMap map, TailCont tc, int most) {
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(clusters * kSplit);
    cfg.blockDim = dim3(NT);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, split_resume<MT, NT, VPT, DVU, MINB>, g, p, syn, out,
                              counter, map, tc, most);
}

template <typename MT, int NT, int VPT, int DVU, int MINB>
SplitKernel split_entry() {
    SplitKernel k;
    k.msg_fp16 = sizeof(MT) == 2;
    k.threads = NT;
    k.vpt = VPT;
    k.dv = DVU;
    k.fn = (const void *)split_resume<MT, NT, VPT, DVU, MINB>;
    k.launch = &launch_split<MT, NT, VPT, DVU, MINB>;
    return k;
}

}  // namespace

void split_table(const SplitKernel **out, int *n) {
    // per precision: the first entry whose blocks hold their faults.  Gross code, 17 and 42
    // resumed shots: 256 x 4 24.0 and 28.3 ms, 384 x 3 25.4 and 33.0, 512 x 2 22.8 and 31.2.
    static const SplitKernel table[] = {
        split_entry<float, 256, 1, 3, 2>(),  split_entry<float, 256, 4, 3, 2>(),
        split_entry<float, 512, 5, 3, 1>(),  split_entry<__half, 256, 1, 3, 2>(),
        split_entry<__half, 256, 4, 3, 2>(), split_entry<__half, 512, 5, 3, 1>(),
    };
    *out = table;
    *n = (int)(sizeof(table) / sizeof(table[0]));
}

}  // namespace qldpc
