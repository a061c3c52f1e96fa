// Fused persistent Relay-BP kernel (paper Sec. 2.3 "Relay decoding", App. A.3).
//
// One thread block decodes one syndrome at a time and pulls the next one from a
// global work counter when it finishes (per-shot early exit, no idle blocks
// behind slow shots).  Per shot:
//   * every edge's message lives in shared memory in one slot, overwritten in
//     place: the check pass turns nu(t-1) into mu(t), the fault pass turns mu(t)
//     into nu(t).  The DC slots of a check are contiguous (128-bit loads and
//     stores in the check pass), with their order inside the check XOR-swizzled
//     by the check index so that the fault pass's gathers and scatters over
//     consecutive checks fall into distinct banks;
//   * the per-fault state (Lambda_j, (1-gamma_j) lambda_j(0), gamma_j) lives in
//     registers: fault j belongs to thread j mod NT for the whole shot;
//   * decisions F_j = [Lambda_j < 0] are sign bits; the warps that decided any fault
//     write them to a bitmap and flip their checks in sigma + H F, which is 0 when
//     the decision explains the syndrome.
// All float arithmetic rounds every + and * separately (__fadd_rn/__fmul_rn), in
// the same order as the single-precision oracle, so results are bit-identical.
//
// This translation unit is compiled once per (message precision, max check
// degree DC, max fault degree DV), selected by QL_MSG_F16, QL_DC and QL_DV.
#include "relay_device.cuh"

#ifndef QL_MSG_F16
#define QL_MSG_F16 0
#endif
#ifndef QL_DC
#define QL_DC 8
#endif
#ifndef QL_DV
#define QL_DV 4
#endif

namespace qldpc {
namespace {

// Block-wide state of the shot in flight, in shared memory: the passes need nearly every
// register of the persistent shapes, and this is read and written at leg boundaries only
// (in registers it cost the passes 600 of 5,850 warp-instructions an iteration, in values
// computed again; gross code, 30,000 shots at 384 threads: 1.77 -> 1.71 ms without).
// A value that changes at a boundary has two copies, used in turn, so that the thread that
// writes the next one never meets a reader of the last one between the same two barriers.
struct ShotState {
    int shot, rec;       // the shot, and its record when it is resumed
    int slot;            // record taken for a suspension (-1: go on)
    long long iters[2];  // iterations run before leg r: iters[r & 1]
    long long wacc[2];   // weight of the new solution, added up by its faults' threads
    long long best[2];   // weight of the kept solution (kNoWeight: none); copy in use: as wacc
};
// Shapes with registers to spare at their launch bounds' residency keep the slot records of
// their faults there: it takes a load's latency out of every fault pass, which shows where
// few warps hide it (8064 faults, 512 x 16, one block per SM: 1.68 -> 1.55 ms).  Giving up a
// resident block for it does not pay (gross code, 256 x 11: 4 blocks 1.05, 3 blocks with the
// records kept 1.15 ms).
template <int NT, int VPT, int MINB>
constexpr bool kKeep = QL_DC == 8 && (65536 / (NT * MINB) / 8 * 8) >= 5 * VPT + 31;
constexpr bool kCut = QL_DC == 8 && !QL_MSG_F16;  // see fault_update
constexpr long long kNoWeight = 0x7fffffffffffffffLL;

// Relay on one shot: the leg schedule around the check and fault passes.  Per
// iteration: check pass | barrier | fault pass | barrier | per-warp convergence
// test.  A leg end adds the weight sum, the next leg's initialisation and one
// barrier.  Called by every thread of the block with block-uniform arguments.
// packed and rb.part: the warp's packed fault slots and the thread's rows with padding, of
// the shot's code; the rest of rb is set here.
// ab selects the copy of st.wacc and st.best in use; the other accumulator is zeroed after
// each use, at least two barriers before it is added into again.  Both start at zero and
// ab persists across the block's shots.
// A solution is kept iff one has been found (sols > 0).
// Tail continuation (TailCont): with tc.mode 1 a shot that reaches a leg boundary after
// tc.cut iterations, with a next leg to run, may be suspended (its state saved in a
// record, no outputs written); RESUME takes the shot of record st.rec up at its boundary.
template <typename MT, int NT, int VPT, int DC, int DV, bool RESUME = false, typename FS>
__device__ __forceinline__ void decode_shot(const FusedGraph &g, const DevParams &p,
                                            const uint64_t *__restrict__ syn, int syn_stride,
                                            int cor_stride, const DecodeOut &out,
                                            unsigned char *msg, uint32_t *fw, uint32_t *fb,
                                            uint32_t *sg, uint32_t *par, ShotState &st, const FS &fs, RowBits &rb,
                                            float (&Lam)[VPT], float (&bb)[VPT],
                                            float (&gg)[VPT], int &ab, const TailCont &tc) {
    const int tid = threadIdx.x;
    const float C = p.clip;
    int leg = 0, sols = 0;
    {
        const uint64_t *sy = syn + (size_t)st.shot * syn_stride;
        load_syndrome<NT>(g, sy, sg);
        row_syndromes<MT, NT>(g, sy, rb);
    }
    if (RESUME) {  // resume at the boundary where the first launch stopped the shot
        const TailRecord r = tc.rec[st.rec];
        leg = r.leg;
        sols = r.sols;
        if (tid == 0) {
            st.iters[leg & 1] = r.iters;
            st.best[ab] = r.have ? r.Wbest : kNoWeight;
        }
        const float *lr = tc.lam + (size_t)st.rec * g.N;
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            const int j = threadIdx.x + q * NT;
            if (j < g.N) Lam[q] = lr[j];
        }
        if (sols > 0) {  // the kept solution, for the same-solution test
            const uint64_t *cor = out.corr + (size_t)st.shot * cor_stride;
            for (int q = tid; q < g.cor_words; q += NT) {
                const uint64_t v = cor[q];
                fb[2 * q] = (uint32_t)v;
                fb[2 * q + 1] = (uint32_t)(v >> 32);
            }
        }
    } else if (tid == 0) {
        st.iters[0] = 0;
        st.best[ab] = kNoWeight;
    }
    // each pass of this loop starts at a leg boundary: the next leg's initial messages, one
    // barrier, the kept solution's update, then the leg's iterations
    uint32_t *pc = par;  // this iteration's parity words: the two buffers take turns
    bool fresh = false, done = false;
    for (;;) {
        if (!done) leg_init<MT, NT, VPT, DV>(g, p, leg, msg, fs, Lam, bb, gg);
        // a long shot with a next leg to run is suspended if a record is free (the next
        // leg's initialisation is redone on resumption from the same state); thread 0
        // decides and takes the record, st.slot tells the block (-1: go on)
        if (!RESUME && tid == 0) {
            int k = -1;
            if (!done && tc.mode == 1 && st.iters[leg & 1] >= tc.cut) {
                const unsigned int c = atomicAdd(tc.count, 1u);
                if (c < (unsigned int)tc.cap) k = (int)c;
            }
            st.slot = k;
        }
        __syncthreads();  // the weight and the leg's initial messages are visible
        if (fresh) {
            const long long W = st.wacc[ab], best = st.best[ab];
            if (W < best)
                keep_solution<NT>(out.corr + (size_t)st.shot * cor_stride, fw, fb, g.cor_words);
            if (tid == 0) {
                st.wacc[ab ^ 1] = 0;
                st.best[ab ^ 1] = W < best ? W : best;
            }
            ab ^= 1;
        }
        if (!RESUME && st.slot >= 0) break;
        if (done) break;
        // iterations this leg may run: its limit and what the budget leaves
        int limit = leg == 0 ? p.T1 : p.T2;
        if (p.max_iters > 0) {
            const long long left = p.max_iters - st.iters[leg & 1];
            limit = left < limit ? (left < 1 ? 1 : (int)left) : limit;
        }
        uint32_t dm;
        bool conv;
        int t = 0;
        do {
            check_pass<NT, DC>(g, reinterpret_cast<MT *>(msg), sg, pc, rb, C);
            __syncthreads();
            dm = fault_pass<MT, NT, VPT, DC, DV, kCut>(g, msg, fw, pc, fs, Lam, bb, gg, C);
            __syncthreads();
            ++t;
            conv = warp_converged(pc, g.m_words);
            pc = pc == par ? par + g.m_words : par;
        } while (!conv && t != limit);
        // a solution equal to the kept one has its weight and cannot replace it
        fresh = conv && !(sols > 0 && warp_same_solution(fw, fb, 2 * g.cor_words));
        if (conv) ++sols;
        if (fresh) add_weight<NT, VPT>(g, dm, st.wacc + ab);
        const long long iters = st.iters[leg & 1] + t;
        done = sols >= p.S || leg == p.R || (p.max_iters > 0 && iters >= p.max_iters);
        if (tid == 0) st.iters[(leg + 1) & 1] = iters;
        ++leg;
    }
    const int slot = RESUME ? -1 : st.slot;  // this shot's last leg boundary set it
    if (slot >= 0) {  // suspended: the state at this boundary; the next leg runs on resumption
        float *lr = tc.lam + (size_t)slot * g.N;
#pragma unroll
        for (int q = 0; q < VPT; ++q) {
            const int j = threadIdx.x + q * NT;
            if (j < g.N) lr[j] = Lam[q];
        }
        if (tid == 0)
            tc.rec[slot] = TailRecord{st.shot, leg, sols, sols > 0 ? 1 : 0, st.iters[leg & 1],
                                      st.best[ab]};
        return;
    }
    if (sols == 0) store_bits<NT>(out.corr + (size_t)st.shot * cor_stride, fw, g.cor_words);
    if (tid == 0) {
        if (out.legs) out.legs[st.shot] = leg;
        if (out.conv) out.conv[st.shot] = sols > 0 ? 1 : 0;
        if (out.iters) out.iters[st.shot] = (int32_t)st.iters[leg & 1];
    }
}

// One block per shot at a time; shots come from a global counter (through the shot
// map's index list when it has one).
// RESUME: the second launch of the tail continuation; shots come from the records of the
// first launch (counter then numbers the records taken), when there are more than `least`.
template <typename MT, int NT, int VPT, int MINB, int DC, int DV, bool RESUME = false>
__global__ void __launch_bounds__(NT, MINB) fused_decode(FusedGraph g, DevParams p,
                                                   const uint64_t *__restrict__ syn, int B,
                                                   DecodeOut out, unsigned int *counter,
                                                   ShotMap map, TailCont tc, int least) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *msg = smem_raw;
    uint32_t *fw, *fb, *sg, *par;
    smem_layout(g, smem_raw, fw, fb, sg, par);
    __shared__ ShotState st;
    // The resuming launch is queued as a programmatic dependent of the first one: its blocks
    // may be placed while the first launch's last shots run, and wait here for its end.
    if (RESUME)
        asm volatile("griddepcontrol.wait;" ::: "memory");
    else
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int limit = RESUME ? (int)min(*tc.count, (unsigned int)tc.cap)
                             : (map.order ? min(*map.count, B) : B);
    if ((int)blockIdx.x >= limit) return;  // as many blocks as shots at most have work
    if (RESUME && limit <= least) return;  // the split launch has taken them
    clear_bitmaps<NT>(g, fw);

    FaultSlots<MT, NT, VPT, kKeep<NT, VPT, MINB>> fs;
    fs.init(g);
    RowBits rb;
    rb.part = setup_rows<MT, NT, DC>(g, msg, p.clip);

    float Lam[VPT], bb[VPT], gg[VPT];
#pragma unroll
    for (int r = 0; r < VPT; ++r) Lam[r] = bb[r] = gg[r] = 0.0f;
    int ab = 0;
    if (threadIdx.x < 2) st.wacc[threadIdx.x] = 0;

    for (;;) {
        __syncthreads();  // the previous shot is done with shared memory and its state
        if (threadIdx.x == 0) {
            const int k = (int)atomicAdd(counter, 1u);
            if (RESUME) {
                st.rec = k;
                st.shot = k < limit ? tc.rec[k].shot : -1;
            } else {
                st.shot = k < limit ? (map.order ? map.order[k] : k) : -1;
            }
        }
        __syncthreads();
        if (st.shot < 0) break;
        decode_shot<MT, NT, VPT, DC, DV, RESUME>(g, p, syn, map.syn_stride, map.cor_stride, out,
                                                 msg, fw, fb, sg, par, st, fs, rb, Lam,
                                                 bb, gg, ab, tc);
    }
}

// Mixed batch: shot b belongs to code code_of_shot[b] of the table; syndromes and
// corrections are rows of fixed strides.  A block re-initialises its shared state
// (padding slots, priors) whenever it moves to a shot of another code.
template <typename MT, int NT, int VPT, int MINB, int DC, int DV>
__global__ void __launch_bounds__(NT, MINB) fused_decode_multi(MultiTable tab,
                                                         const int32_t *__restrict__ code_of_shot,
                                                         const uint64_t *__restrict__ syn,
                                                         int syn_stride, int cor_stride, int B,
                                                         DecodeOut out, unsigned int *counter) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *msg = smem_raw;
    __shared__ FusedGraph s_g;
    __shared__ DevParams s_p;
    __shared__ ShotState st;
    __shared__ int s_code;
    int cur = -1;
    FaultSlots<MT, NT, VPT> fs;
    fs.n = 0;
    fs.records = false;
    RowBits rb;
    rb.part = 0u;

    float Lam[VPT], bb[VPT], gg[VPT];
#pragma unroll
    for (int r = 0; r < VPT; ++r) Lam[r] = bb[r] = gg[r] = 0.0f;
    int ab = 0;
    if (threadIdx.x < 2) st.wacc[threadIdx.x] = 0;

    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            const int shot = (int)atomicAdd(counter, 1u);
            st.shot = shot;
            int c = shot < B ? code_of_shot[shot] : 0;
            if (c < 0 || c >= tab.n) c = -1;  // invalid code id: the shot is skipped
            s_code = c;
            if (c >= 0 && c != cur) {
                s_g = tab.g[c];
                s_p = tab.p[c];
            }
        }
        __syncthreads();
        const int shot = st.shot, code = s_code;
        if (shot >= B) break;
        if (code < 0) {  // not a code of the table: marked by iters = -1
            if (threadIdx.x == 0) {
                if (out.legs) out.legs[shot] = 0;
                if (out.conv) out.conv[shot] = 0;
                if (out.iters) out.iters[shot] = -1;
            }
            continue;
        }
        uint32_t *fw, *fb, *sg, *par;
            smem_layout(s_g, smem_raw, fw, fb, sg, par);
        if (code != cur) {
            clear_bitmaps<NT>(s_g, fw);
            fs.init(s_g);
            rb.part = setup_rows<MT, NT, DC>(s_g, msg, s_p.clip);
            cur = code;
            __syncthreads();
        }
        decode_shot<MT, NT, VPT, DC, DV>(s_g, s_p, syn, syn_stride, cor_stride, out, msg, fw, fb,
                                         sg, par, st, fs, rb, Lam, bb, gg, ab,
                                         TailCont{});
    }
}

// First leg without early exit, every iteration recorded (one shot per block).
template <typename MT, int NT, int VPT, int DC, int DV>
__global__ void __launch_bounds__(NT) fused_trace(FusedGraph g, DevParams p,
                                                  const uint64_t *__restrict__ syn, int B, int T,
                                                  int E, float *marg, float *nu, float *mu) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *msg = smem_raw;
    uint32_t *fw, *fb, *sg, *par;
    smem_layout(g, smem_raw, fw, fb, sg, par);
    const int shot = blockIdx.x;
    const float C = p.clip;
    clear_bitmaps<NT>(g, fw);
    load_syndrome<NT>(g, syn + (size_t)shot * g.syn_words, sg);
    float Lam[VPT], bb[VPT], gg[VPT];
#pragma unroll
    for (int r = 0; r < VPT; ++r) Lam[r] = bb[r] = gg[r] = 0.0f;
    FaultSlots<MT, NT, VPT> fs;
    fs.init(g);
    RowBits rb;
    rb.part = setup_rows<MT, NT, DC>(g, msg, p.clip);
    row_syndromes<MT, NT>(g, syn + (size_t)shot * g.syn_words, rb);
    __syncthreads();
    leg_init<MT, NT, VPT, DV>(g, p, 0, msg, fs, Lam, bb, gg);
    __syncthreads();
    const int nslots = g.msg_bytes / (int)sizeof(MT);
    for (int t = 0; t < T; ++t) {
        const size_t o = (size_t)t * B + shot;
        check_pass<NT, DC>(g, reinterpret_cast<MT *>(msg), sg, par, rb, C);
        __syncthreads();
        if (mu)
            for (int s = threadIdx.x; s < nslots; s += NT) {
                const int e = g.slot_edge[s];
                if (e >= 0) mu[o * E + e] = Msg<MT>::ld(msg, s * (int)sizeof(MT));
            }
        __syncthreads();
        fault_pass<MT, NT, VPT, DC, DV>(g, msg, fw, par, fs, Lam, bb, gg, C);
        __syncthreads();
        if (marg) {
#pragma unroll
            for (int r = 0; r < VPT; ++r) {
                const int j = threadIdx.x + r * NT;
                if (j < g.N) marg[o * g.N + j] = Lam[r];
            }
        }
        if (nu)
            for (int s = threadIdx.x; s < nslots; s += NT) {
                const int e = g.slot_edge[s];
                if (e < 0) continue;
                const float x = Msg<MT>::ld(msg, s * (int)sizeof(MT));  // stored unclamped
                nu[o * E + e] = fabsf(x) > C ? copysignf(C, x) : x;
            }
        __syncthreads();
    }
}

template <typename MT, int NT, int VPT, int MINB, int DC, int DV, bool RESUME>
cudaError_t launch_decode(dim3 grid, size_t smem, cudaStream_t st, const FusedGraph &g,
                          const DevParams &p, const uint64_t *syn, int B, DecodeOut out,
                          unsigned int *counter, ShotMap map, TailCont tc, int least) {
    if (RESUME) {  // without work it costs a call 1 us behind the first launch, not 5
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = grid;
        cfg.blockDim = dim3(NT);
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, fused_decode<MT, NT, VPT, MINB, DC, DV, RESUME>, g, p, syn,
                                  B, out, counter, map, tc, least);
    }
    fused_decode<MT, NT, VPT, MINB, DC, DV, RESUME><<<grid, NT, smem, st>>>(g, p, syn, B, out,
                                                                            counter, map, tc, least);
    return cudaGetLastError();
}

template <typename MT, int NT, int VPT, int MINB, int DC, int DV>
cudaError_t launch_multi(dim3 grid, size_t smem, cudaStream_t st, const MultiTable &tab,
                         const int32_t *code_of_shot, const uint64_t *syn, int syn_stride,
                         int cor_stride, int B, DecodeOut out, unsigned int *counter) {
    fused_decode_multi<MT, NT, VPT, MINB, DC, DV><<<grid, NT, smem, st>>>(
        tab, code_of_shot, syn, syn_stride, cor_stride, B, out, counter);
    return cudaGetLastError();
}

template <typename MT, int NT, int VPT, int DC, int DV>
cudaError_t launch_trace(dim3 grid, size_t smem, cudaStream_t st, const FusedGraph &g,
                         const DevParams &p, const uint64_t *syn, int B, int T, float *marg,
                         float *nu, float *mu) {
    fused_trace<MT, NT, VPT, DC, DV><<<grid, NT, smem, st>>>(g, p, syn, B, T, g.E, marg, nu, mu);
    return cudaGetLastError();
}

#if QL_MSG_F16
using MsgT = __half;
#else
using MsgT = float;
#endif

template <int NT, int VPT, int MINB, bool TRACE, int WAVES = 0>
FusedKernel entry() {
    FusedKernel k;
    k.waves = QL_DC == 8 ? WAVES : 0;
    k.msg_fp16 = QL_MSG_F16;
    k.threads = NT;
    k.min_blocks = MINB;
    k.vpt = VPT;
    k.dc = QL_DC;
    k.dv = QL_DV;
    k.decode_fn = (const void *)fused_decode<MsgT, NT, VPT, MINB, QL_DC, QL_DV>;
    k.launch_decode = &launch_decode<MsgT, NT, VPT, MINB, QL_DC, QL_DV, false>;
    if constexpr (NT == 1024) {  // the shapes of the tail continuation's second launch
        k.resume_fn = (const void *)fused_decode<MsgT, NT, VPT, MINB, QL_DC, QL_DV, true>;
        k.launch_resume = &launch_decode<MsgT, NT, VPT, MINB, QL_DC, QL_DV, true>;
    } else {
        k.resume_fn = nullptr;
        k.launch_resume = nullptr;
    }
    k.multi_fn = (const void *)fused_decode_multi<MsgT, NT, VPT, MINB, QL_DC, QL_DV>;
    k.launch_multi = &launch_multi<MsgT, NT, VPT, MINB, QL_DC, QL_DV>;
    if constexpr (TRACE) {
        k.trace_fn = (const void *)fused_trace<MsgT, NT, VPT, QL_DC, QL_DV>;
        k.launch_trace = &launch_trace<MsgT, NT, VPT, QL_DC, QL_DV>;
    } else {
        k.trace_fn = nullptr;
        k.launch_trace = nullptr;
    }
    return k;
}

}  // namespace

#define QL_CAT2(P, DC, DV) fused_table_##P##_##DC##_##DV
#define QL_EXPAND(P, DC, DV) QL_CAT2(P, DC, DV)
#if QL_MSG_F16
#define QL_P f16
#else
#define QL_P f32
#endif

void QL_EXPAND(QL_P, QL_DC, QL_DV)(const FusedKernel **out, int *n) {
    // (threads, faults per thread, min resident blocks): the first entry that holds the graph
    // (threads * vpt >= N) is used unless the caller asks for a block size; the last
    // entry also serves the trace kernel; the 1024-thread entries serve the resuming
    // launch of the tail continuation; the entries with a number of waves serve small batches.
    //
    // Rows of up to 8 slots: the blocks are narrow, with as many faults per thread as the
    // registers hold at full residency, since the cost of an iteration that does not depend
    // on the faults (barriers, the convergence test, the check pass's uneven rows) is per
    // warp.  The reaches are chosen so that the detector models of the three codes fill all
    // fault slots but the last at most of their usual numbers of rounds (each_fault; counted, no
    // warp does for the 72-qubit code at 2, 3, 5, 9, 14, 15 and 18 rounds, the 144-qubit code at 0,
    // 1, 2, 7 and 16, the 288-qubit code at 0, 3, 4, 11, 13, 16 and 17).  Measured, old shape ->
    // this one: 72 faults 256 x 4 -> 32 x 3 2.26 -> 0.59 ms (60,000 shots), 720 faults 256 x 4 ->
    // 64 x 12 1.13 -> 0.75 ms, gross code 512 x 6 -> 256 x 11 1.88 -> 1.59 ms (30,000), 8064 faults
    // 1024 x 8 -> 256 x 32 1.72 -> 1.49 ms (8,000).
    static const FusedKernel table[] = {
#if QL_DC == 8
        entry<32, 3, 32, false>(),
        entry<64, 4, 16, false, 3>(),
        entry<64, 8, 16, false>(),
        entry<64, 12, 16, false>(),
        entry<64, 13, 12, false>(),
        entry<128, 8, 8, false>(),
#endif
        entry<256, 4, 4, false, 12>(),
#if QL_DC == 8
        entry<128, 10, 6, false>(),
        entry<128, 12, 6, false>(),
        entry<128, 15, 5, false>(),
        entry<128, 18, 5, false>(),
        entry<256, 10, 4, false>(),
        entry<256, 11, 4, false>(),
        entry<256, 12, 4, false>(),
#endif
        entry<512, 6, 2, false, 2>(),
#if QL_DC != 8
        entry<256, 12, 4, false>(),
#endif
        entry<384, 8, 3, false>(),
        entry<640, 5, 2, false>(),
        entry<768, 4, 2, false>(),
        entry<1024, 3, 1, false>(),
#if QL_DC == 8
        entry<256, 14, 3, false>(),
        entry<256, 16, 3, false>(),
        entry<256, 18, 3, false>(),
        entry<256, 22, 2, false>(),
        entry<256, 25, 2, false>(),
        entry<384, 18, 2, false>(),
        entry<256, 32, 2, false>(),
#endif
        entry<1024, 8, 1, false, 2>(),
        entry<512, 16, 1, false>(),
        entry<512, 32, 1, true>(),
    };
    *out = table;
    *n = (int)(sizeof(table) / sizeof(table[0]));
}

}  // namespace qldpc
