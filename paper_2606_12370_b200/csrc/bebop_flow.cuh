// The stream: bebop_verify (with its TV output) and bebop_tv as a stream of logits through a cluster of CTAs, one CTA per SM.
//
// A unit is a row pair (target row k, draft row k of a sequence) or a sequence's bonus row.  Every cluster owns a contiguous
// run of the call's units, weighed by their rows, and each of its CTAs has one slice of every row of the run: no tickets, and no
// waiting on another cluster.  A unit goes through twice,
//   pass 1  per chunk of 256 (short rows: 128) 16-byte vectors, a warp each: the reference exponent E (an integer) and the sum of
//           e = 2^(x c - E);
//   pass 2  per half as many vectors of both rows: the residuals r' = max(0, e_p - rho e_q) = (p - q) S_p, rho = S_p / S_q,
// and the stream interleaves them, pass 1 of unit u before pass 2 of unit u - 1 (small chunks: u - 2 or u - 3): between the passes of a unit lies
// another unit's work, under which the exchange of the sums within the cluster disappears, and the second pass finds its logits in L2
// (two units of every cluster are under way, 90 MB in all at 151,936 bf16 logits; DRAM reads 1.07 times the logits of 256 such sequences, K = 3, 1.01
// of 64), or, if the rows are short, in the stage where pass 1 left them (FlowResident).
//
// Warps: the consumers; a producer (one thread: bulk copies into a ring of 192 KB in three to eight stages, with a description
// each); one or two warps that exchange and merge the sums of pass 1, one that writes out the masses of pass 2, and a finisher.  The
// consumers do not meet: a warp takes the chunk of a stage that falls to it (the first chunk's warp moves on from
// stage to stage, so that short stages load the warps evenly), leaves its sums in a table and moves on.  The exchange warp adds
// the chunks up, half a warp per row, sends the CTA's sums to the cluster through distributed shared memory, merges what it is
// sent (exact powers of two, one fixed order, the same bits in every CTA) and hands the consumers rho.  The CTA that
// delivers the last part of a sequence has its finisher complete it -- accept scan (Algorithm 3), TV, the fast draw with its
// certificate or a place in the list for the fp64 re-draw -- while the stream goes on.
//
// What bounds it: the exponential unit, 16 lanes per SM and clock, which two passes keep for 104 us of the 150 that 768 row pairs of
// 151,936 bf16 logits take; 69 per cent busy while an SM works (6.2 instructions per logit and pass), the rest are the chains at
// both ends of a warp's chunk (barrier, maximum, reduction) and the ends of the clusters' runs.  Neither DRAM nor L2 does (the
// bulk copies reach 19 TB/s out of L2).  What a task costs beyond its exponentials, 0.3 to 0.4 us, hardly depends on its size:
// 768 row pairs in stages of 32, 48, 64 KB 182, 164, 152 us; sixteen warps of eight vectors a lane are better than twelve (172) or than
// 24 of four (164), except on short rows, whose units those pieces fit better.  The same calls through the kernels in
// whose place the stream stands (exponentials parked in tensor memory; two full sweeps over DRAM): 768 row pairs 168 us, 256
// sequences of 151,936, K = 3, 198 (178), 1,024 of them, K = 4 ragged, 686 (531), 192 of 32,000, K = 7 ragged, 83 (60.5).
// The size of the consumers' loop counts: a branch in it for the bonus row's masses cost 2 to 7 per cent, a call in its place 6 (their sums
// are exact for all rows instead), a vote in front of the load of a task's description 1.  Tried and left out: more and smaller stages for
// short rows (1,000 of 8,000, K = 8, 174 us in four stages of 48 KB, 191 in twelve of 16), one place in the producer that hands out all tasks
// (256 of 151,936 178 -> 183 us), the finisher's loads all asked for at once (no change, and short rows 5 per cent slower), warps in two or four groups on alternate stages (179 us and 196 for the 256 sequences), two or three units
// between the passes (184), four CTAs a cluster (209 to 222).
//
// Every wait is bounded; one that gives up sets the wait flag and the CTA's abort flag, under which all warps run out.  No
// multicast; copies from this GPU's own memory only.
#pragma once
#include "bebop_chunk.cuh"

namespace bebop {

extern cudaEvent_t g_ev_start, g_ev_stop;

namespace {

// Consumer warps; vectors per lane of a chunk; units under way at most (tables by the unit's number mod LSL); exchange warps; RES: a
// unit's logits stay in their stage until pass 2, which then needs no second copy.
template <int W, int Q, int SL, int X, bool RES> struct FlowDims {
    static constexpr int LW = W, LQV = Q, LSL = SL, LNX = X;
    static constexpr bool LRES = RES;
    static constexpr int LCV = 32 * Q;                       // vectors of a chunk of pass 1; a chunk of pass 2 has half as many of each row
    static constexpr int LRING = 196608, LSTAGE = W * LCV * 16, LNS = RES ? 8 : LRING / LSTAGE;      // (RES: so many stages at most, of the size of a unit)
    static constexpr int W_FPROD = W, W_PUB = W + 1, W_FIN = W + 2, W_EXCH = W + 3, LT = (W + 3 + X) * 32;
    static constexpr int MAXCH = RES ? W / 2 : (Q == 8 ? 20480 : 12288) / LCV;         // chunks of a row slice, at most
};
constexpr int LUD = 16, LMB = 256;              // unit descriptions in flight, entries of the finisher's mailbox
// Long: rows of which a CTA's slice is long enough for large chunks, which cost less per logit; Short: finer pieces for short rows.
// Resident: rows so short that four units or more fit the ring.  Their units are over sooner than one producer thread hands out
// three tasks, or one warp exchanges their sums: 1,000 sequences of 8,000 bf16 logits, K = 8, 178 us as Short (whose producer was busy for 324 of
// 349 us of 2,000 such, its exchange warp for 271), 159 with both rows' pass 1 in one task, 145 with the logits kept, 131 with two
// exchange warps; 2,000 of 11,000, K = 3, 194 -> 134, 1,000 of 5,000 fp32, K = 8, 149 -> 107.
using FlowLong = FlowDims<16, 8, 2, 1, false>;
using FlowShort = FlowDims<24, 4, 4, 1, false>;
using FlowResident = FlowDims<24, 4, 4, 2, true>;
constexpr int kResidentVecs = FlowResident::MAXCH * FlowResident::LCV;     // of a row, at most
constexpr uint32_t kLSpin = 1u << 20;
constexpr int kFailed = 1 << 30;              // mark in a sequence's count: given up, its outputs say so

struct FlowRow { double inv_s, ub; int e, st; double pad; };         // a merged row: 1/S, bound of sum p^2, exponent, status
struct FlowRec { double s, ub; int e, bad; double pad; };              // a CTA's part of a row
struct __align__(16) FlowUnit {
    int b, k, kind, unit;                      // b < 0: no more units; kind: bit 0 a row pair (else the bonus row), above it the sequence's length
    __device__ __forceinline__ bool pair() const { return kind & 1; }
};
struct __align__(16) FlowSrc { const char *p, *q; };                   // the CTA's slices of a unit's rows (no q: a bonus row)

struct FlowArgs {
    RowArgs r;
    const int32_t* draft_tokens;
    const float* u_accept;
    const float* u_final;
    VerifyOut o;
    float* s_aux;
    int share;                                // rows of a cluster, at most; 0: even shares; -1: even shares of ragged sequences
    int lag;                                  // units between a unit's passes, below LSL
    int ns, pitch;                            // resident form: stages, bytes of one
    int C, G, nch, sv;                        // CTAs per cluster, clusters, chunks and vectors of a row slice
    int expire;                               // test hook: the helper's wait for the cluster's sums counts as run out
    float kappa;
    int* wait_failed;
    unsigned long long* fb_count;
    FbRec* fb_list;
    int* seqcnt;                              // [B] parts of the sequence delivered
    FlowRow* rows;                            // [units][2]
    double* smass;                            // [units][C] mass of a slice
    double* sauxp;                            // [units][C] bebop_tv: sum of q over the tokens with q <= p
    double* mass;                             // [units][C][2 nch] mass of a chunk (row pair: of pass 2; bonus row: of pass 1)
};

template <class F> struct FlowShared {
    unsigned long long full[F::LNS], empty[F::LNS];
    unsigned long long ud[LUD];               // a unit's description is there
    unsigned long long p1[F::LSL], p2[F::LSL];      // by slot of the unit: all consumer warps are through with its pass 1 / pass 2
    unsigned long long rec[F::LSL];                // ... the cluster's records of its rows are there
    unsigned long long stat[F::LSL];               // ... its rows are merged
    unsigned long long pub[F::LSL];                // ... the sums of its pass 2 have been read
    int4 task[F::LNS];
    FlowUnit unit[LUD];
    FlowSrc src[LUD];
    float uc[LUD];                            // log2(e) / tau of the unit's sequence
    float4 scale[F::LSL];                          // exponents of both rows, rho as two floats
    double inv[F::LSL][2];                         // 1/S of both rows
    FlowRec rrec[F::LSL][kFlowMaxCluster][2];
    int4 part[F::LSL][2][F::MAXCH];          // chunks of pass 1: warp_sum_words, exponent, upper bound of the sum of e^2 in 2^-15
    int2 cm[F::LSL][2 * F::MAXCH], ca[F::LSL][2 * F::MAXCH];
    int wsum[F::LT / 32];
    int start_b, start_k, end_w, start_w;     // the cluster's run of units: the first one, weights of its begin and end
    int mbox[LMB], mb_tail, mb_head, mb_done;
    int abort;
};

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ bool mbar_try_cluster(uint32_t addr, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void mbar_arrive_remote(uint32_t a) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" :: "r"(a) : "memory");
}
__device__ __forceinline__ void bulk_load_hint(uint32_t dst, const void* src, uint32_t bytes, unsigned long long* bar, unsigned long long policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy) : "memory");
}
// What the call clears (the sequences' counts, the re-draw's list and counters, the wait flag) is clear from here on.  Everything
// else goes ahead of it: the clearing kernel in front has waited for what came before the call.
__device__ __forceinline__ void flow_cleared() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <class F> __device__ __forceinline__ void flow_give_up(const FlowArgs& a, FlowShared<F>& S) {
    flow_cleared();
    atomicExch(a.wait_failed, 1);
    *(volatile int*)&S.abort = 1;
}
// bounded; gives up at once when the CTA has given up somewhere; the answer is the lane's own
template <class F> __device__ __noinline__ bool flow_wait_slow(const FlowArgs& a, FlowShared<F>& S, uint32_t addr, uint32_t parity) {
    for (uint32_t i = 0; i < kLSpin; ++i) {
        if (mbar_try(addr, parity)) return true;
        if (*(volatile int*)&S.abort) return false;
    }
    flow_give_up(a, S);
    return false;
}
template <class F> __device__ __forceinline__ bool flow_wait_one(const FlowArgs& a, FlowShared<F>& S, unsigned long long* b, uint32_t parity) {
    const uint32_t addr = smem_u32(b);
    return mbar_try(addr, parity) || flow_wait_slow(a, S, addr, parity);
}
// The same for a whole warp, with one answer for all of its lanes: a lane that gave up alone would leave the others in warp-wide
// reductions that it never comes to.
template <bool CL, class F> __device__ __noinline__ bool flow_wait_slow_warp(const FlowArgs& a, FlowShared<F>& S, uint32_t addr, uint32_t parity) {
    for (uint32_t i = 0; i < kLSpin; ++i) {
        if (__all_sync(0xffffffffu, CL ? mbar_try_cluster(addr, parity) : mbar_try(addr, parity))) return true;
        if (__any_sync(0xffffffffu, *(volatile int*)&S.abort)) return false;
    }
    flow_give_up(a, S);
    return false;
}
template <bool CL = false, class F> __device__ __forceinline__ bool flow_wait(const FlowArgs& a, FlowShared<F>& S, unsigned long long* b, uint32_t parity) {
    const uint32_t addr = smem_u32(b);
    if (__all_sync(0xffffffffu, CL ? mbar_try_cluster(addr, parity) : mbar_try(addr, parity))) return true;
    return flow_wait_slow_warp<CL>(a, S, addr, parity);
}

// ------------------------------------------------------------------ the cluster's run of units
// From one share's begin to the next, where every sequence weighs w: `share` rows on, or one less where a row pair would be cut
// (units begin at even places of a sequence).
__host__ __device__ __forceinline__ void flow_next(int& at, int& r, int share, int step, int w) {
    at += share; r += step;
    if (r >= w) r -= w;
    if (r & 1) { --r; --at; }
}
// A sequence weighs 2 L + 1 rows (bebop_tv: 2), in order; cluster g takes the units that begin in its share of the weight.
template <bool TVM, class F>
__device__ __forceinline__ void flow_share(const FlowArgs& a, FlowShared<F>& S, int g) {
    const RowArgs& R = a.r;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (a.share >= 0) {                                     // sequences of one weight
        if (tid == 0) {
            const int w = TVM ? 2 : 2 * R.K + 1, total = R.B * w;
            int at = 0, r = 0;                              // where the run begins, and how far inside its sequence
            if (a.share > 0) {                              // every cluster takes what fits its share
                const int step = a.share % w;
                for (int i = 0; i < g; ++i) flow_next(at, r, a.share, step, w);
                S.start_b = at / w; S.start_k = r / 2; S.start_w = at;
                flow_next(at, r, a.share, step, w);
                S.end_w = min(at, total);
            } else {                                        // the first unit that begins at the run's even share or later
                const int lo = (int)((long long)total * g / a.G), k = (lo % w + 1) / 2;
                S.start_b = lo / w + (TVM ? k : 0); S.start_k = TVM ? 0 : k; S.start_w = lo - lo % w + 2 * k;
                S.end_w = (int)((long long)total * (g + 1) / a.G);
            }
        }
        return;
    }
    const int seg = (R.B + F::LT - 1) / F::LT, b0 = min(tid * seg, R.B), b1 = min(b0 + seg, R.B);
    int mine = 0;
    for (int b = b0; b < b1; ++b) mine += TVM ? 2 : 2 * len_of(R, b) + 1;
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const int t = __shfl_up_sync(0xffffffffu, incl, o); if (lane >= o) incl += t; }
    if (lane == 31) S.wsum[warp] = incl;
    __syncthreads();
    int below = 0, total = 0;
    for (int w = 0; w < F::LT / 32; ++w) { const int x = S.wsum[w]; if (w < warp) below += x; total += x; }
    const int lo = (int)((long long)total * g / a.G), hi = (int)((long long)total * (g + 1) / a.G);
    if (tid == 0) S.end_w = hi;                             // (where lo == hi, start_b = B: no units)
    // the first unit that begins at lo or later
    int at = below + incl - mine;
    if (lo < hi && at + mine > lo && at <= lo) {
        // (the unit that begins here may be the next sequence's first)
        int b = b0, k = 0;
        while (at < lo) {
            const int L = TVM ? 1 : len_of(R, b);
            at += k < L ? 2 : 1;
            if (++k > (TVM ? 0 : L)) { ++b; k = 0; }
        }
        S.start_b = b; S.start_k = k; S.start_w = at;
    }
}

// ------------------------------------------------------------------ producer
// One thread, whose instructions are its time (some ten cycles each beside the consumers): what does not change from unit to unit is
// worked out once, rows are found by adding strides, and pass 2 finds its rows where pass 1 left them.
template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_producer(const FlowArgs& a, FlowShared<F>& S, unsigned char* ring, int rank) {
    constexpr int VEC = Elem<DT>::VEC, CV = F::LCV / 2;
    const RowArgs& R = a.r;
    const int v0 = rank * a.sv, nv = max(min(a.sv, R.nvec - v0), 0);
    const int ragged = (R.V % VEC != 0 && nv > 0 && v0 + nv == R.nvec) ? 1 << 16 : 0;
    unsigned long long keep, drop;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(drop));
    int st = 0, n = 0, rot = 0;                              // stage, tasks, warp of the next task's first chunk
    uint32_t ph = 1;                                        // parity the stage's `empty` must have completed
    bool ok = true;
    // task: x = kind (0 pass 1, 1 pass 2, 3 stop) | row << 2 | last << 3 | first warp << 4 | chunks << 10 | first chunk << 16;
    // y = vectors of the task (of one row) | ragged << 16, z = c, w = unit's number
    auto issue = [&](int x, int chunks, int y, float c, uint32_t u, const char* src0, const char* src1, unsigned long long pol) {
        if (!flow_wait_one(a, S, &S.empty[st], ph)) { ok = false; return; }
        S.task[st] = make_int4(x | rot << 4 | chunks << 10, y, __float_as_int(c), (int)u);
        const uint32_t bytes = (uint32_t)(y & 0xffff) * 16u, dst = smem_u32(ring + (size_t)st * F::LSTAGE);
        if (bytes) {
            mbar_arrive_expect(&S.full[st], src1 ? 2u * bytes : bytes);
            bulk_load_hint(dst, src0, bytes, &S.full[st], pol);
            if (src1) bulk_load_hint(dst + F::LSTAGE / 2, src1, bytes, &S.full[st], pol);
        } else mbar_arrive(&S.full[st]);
        rot += chunks; if (rot >= F::LW) rot -= F::LW;
        ++n;
        if (++st == F::LNS) { st = 0; ph ^= 1u; }
    };
    auto pass1 = [&](const char* row, int which, bool end, float c, uint32_t u, unsigned long long pol) {
        int c0 = 0, left = nv;
        do {
            const int vecs = min(left, F::LW * F::LCV);
            left -= vecs;
            issue(which << 2 | (end && left == 0 ? 8 : 0) | c0 << 16, (vecs + F::LCV - 1) / F::LCV, vecs | (left == 0 ? ragged : 0), c, u, row, nullptr, pol);
            c0 += F::LW; row += F::LW * F::LCV * 16;
        } while (ok && left > 0);
    };
    auto pass2 = [&](uint32_t u) {
        const FlowSrc x = S.src[u % LUD];
        const float c = S.uc[u % LUD];
        if (!x.q || nv == 0) { issue(1 | 8, 0, 0, c, u, nullptr, nullptr, drop); return; }
        const char *p = x.p, *q = x.q;
        int c0 = 0, left = nv;
        do {
            const int vecs = min(left, F::LW * CV);
            left -= vecs;
            issue(1 | (left == 0 ? 8 : 0) | c0 << 16, (vecs + CV - 1) / CV, vecs | (left == 0 ? ragged : 0), c, u, p, q, drop);
            c0 += F::LW; p += F::LW * CV * 16; q += F::LW * CV * 16;
        } while (ok && left > 0);
    };
    int b = S.start_b, k = S.start_k, w = S.start_w;
    uint32_t u = 0;
    const char* seq_p = R.target + (int64_t)b * R.t_seq_rows * R.t_row_bytes + (int64_t)v0 * 16;          // the sequence's first rows, at this CTA's slice
    const char* seq_q = R.draft + (int64_t)b * R.d_seq_rows * R.d_row_bytes + (int64_t)v0 * 16;
    const char *p = seq_p + k * R.t_row_bytes, *q = seq_q + k * R.d_row_bytes;
    const int64_t seq_p_bytes = R.t_seq_rows * R.t_row_bytes, seq_q_bytes = R.d_seq_rows * R.d_row_bytes;
    // a sequence's length and temperature are asked for one sequence ahead
    auto len = [&](int i) { return TVM ? 1 : len_of(R, min(i, R.B - 1)); };
    int L = len(b), L1 = len(b + 1);
    float tau1 = tau_of(R, min(b + 1, R.B - 1)), c = temp_scale(tau_of(R, min(b, R.B - 1))).hi;
    while (ok && w < S.end_w && b < R.B) {
        const bool pair = k < L;
        FlowUnit x;
        x.b = b; x.k = k; x.kind = 2 * L + (pair ? 1 : 0); x.unit = TVM ? b : b * (R.K + 1) + k;
        S.unit[u % LUD] = x;
        S.uc[u % LUD] = c;
        mbar_arrive(&S.ud[u % LUD]);
        FlowSrc y; y.p = p; y.q = pair ? q : nullptr;
        S.src[u % LUD] = y;
        if (!pair) pass1(p, 0, true, c, u, drop);
        else {
            pass1(p, 0, false, c, u, keep);
            if (ok) pass1(q, 1, true, c, u, keep);
        }
        if (ok && u >= (uint32_t)a.lag) pass2(u - a.lag);
        ++u;
        w += pair ? 2 : 1;
        p += R.t_row_bytes; q += R.d_row_bytes;
        if (++k > (TVM ? 0 : L)) {
            ++b; k = 0;
            seq_p += seq_p_bytes; seq_q += seq_q_bytes;
            p = seq_p; q = seq_q;
            L = L1; c = temp_scale(tau1).hi;
            L1 = len(b + 1); tau1 = tau_of(R, min(b + 1, R.B - 1));
        }
    }
    for (uint32_t i = u < (uint32_t)a.lag ? 0u : u - a.lag; ok && i < u; ++i) pass2(i);
    for (int i = 0; i < F::LNX; ++i) { S.unit[(u + i) % LUD].b = -1; mbar_arrive(&S.ud[(u + i) % LUD]); }          // (an end for each exchange warp)
    if (ok) issue(3, 0, 0, 0.f, u, nullptr, nullptr, drop);
    // no copy of this CTA is under way when it leaves: the last ones have arrived (bounded)
    for (int i = 0; i < F::LNS && i < n; ++i) {
        if (--st < 0) { st = F::LNS - 1; ph ^= 1u; }
        for (uint32_t t = 0; t < kLSpin && !mbar_try(smem_u32(&S.full[st]), ph ^ 1u); ++t) {}
    }
}

// The producer of the resident form: a unit is one task and stays in its stage through both passes.
template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_producer_res(const FlowArgs& a, FlowShared<F>& S, unsigned char* ring, int rank) {
    constexpr int VEC = Elem<DT>::VEC, CV = F::LCV / 2;
    const RowArgs& R = a.r;
    const int v0 = rank * a.sv, nv = max(min(a.sv, R.nvec - v0), 0), n1 = (nv + F::LCV - 1) / F::LCV, n2 = (nv + CV - 1) / CV;
    const int y = nv | (R.V % VEC != 0 && nv > 0 && v0 + nv == R.nvec ? 1 << 16 : 0);
    int st = 0, n = 0, rot = 0;
    uint32_t ph = 1, u = 0;
    int b = S.start_b, k = S.start_k, w = S.start_w;
    const char* p = R.target + ((int64_t)b * R.t_seq_rows + k) * R.t_row_bytes + (int64_t)v0 * 16;
    const char* q = R.draft + ((int64_t)b * R.d_seq_rows + k) * R.d_row_bytes + (int64_t)v0 * 16;
    auto len = [&](int i) { return TVM ? 1 : len_of(R, min(i, R.B - 1)); };
    int L = len(b), L1 = len(b + 1);
    float tau1 = tau_of(R, min(b + 1, R.B - 1)), c = temp_scale(tau_of(R, min(b, R.B - 1))).hi;
    bool ok = true;
    for (;;) {
        // task: x = stop (3) | row pair << 2 | first warp of pass 1 << 4 | its chunks << 10 | first warp of pass 2 << 16 | its chunks << 22;
        // y = vectors of a row | ragged << 16, z = c, w = unit's number
        const bool more = w < S.end_w && b < R.B, pair = more && k < L;
        if (!flow_wait_one(a, S, &S.empty[st], ph)) { ok = false; break; }
        if (!more) break;
        FlowUnit x;
        x.b = b; x.k = k; x.kind = 2 * L + (pair ? 1 : 0); x.unit = TVM ? b : b * (R.K + 1) + k;
        S.unit[u % LUD] = x;
        mbar_arrive(&S.ud[u % LUD]);
        int t = rot << 4;
        const int chunks = pair ? 2 * n1 : n1;
        rot += chunks; if (rot >= F::LW) rot -= F::LW;
        t |= chunks << 10 | rot << 16;
        if (pair) { t |= 4 | n2 << 22; rot += n2; if (rot >= F::LW) rot -= F::LW; }
        S.task[st] = make_int4(t, y, __float_as_int(c), (int)u);
        const uint32_t bytes = (uint32_t)nv * 16u, dst = smem_u32(ring) + (uint32_t)(st * a.pitch);
        if (bytes) {
            mbar_arrive_expect(&S.full[st], pair ? 2u * bytes : bytes);
            bulk_load(dst, p, bytes, &S.full[st]);
            if (pair) bulk_load(dst + a.pitch / 2, q, bytes, &S.full[st]);
        } else mbar_arrive(&S.full[st]);
        ++n; ++u;
        if (++st == a.ns) { st = 0; ph ^= 1u; }
        w += pair ? 2 : 1;
        p += R.t_row_bytes; q += R.d_row_bytes;
        if (++k > (TVM ? 0 : L)) {
            ++b; k = 0;
            p = R.target + (int64_t)b * R.t_seq_rows * R.t_row_bytes + (int64_t)v0 * 16;
            q = R.draft + (int64_t)b * R.d_seq_rows * R.d_row_bytes + (int64_t)v0 * 16;
            L = L1; c = temp_scale(tau1).hi;
            L1 = len(b + 1); tau1 = tau_of(R, min(b + 1, R.B - 1));
        }
    }
    for (int i = 0; i < F::LNX; ++i) { S.unit[(u + i) % LUD].b = -1; mbar_arrive(&S.ud[(u + i) % LUD]); }          // (an end for each exchange warp)
    if (ok) {
        S.task[st] = make_int4(3, 0, 0, (int)u);
        mbar_arrive(&S.full[st]);
        ++n;
        if (++st == a.ns) { st = 0; ph ^= 1u; }
    }
    // no copy of this CTA is under way when it leaves: the last ones have arrived (bounded)
    for (int i = 0; i < a.ns && i < n; ++i) {
        if (--st < 0) { st = a.ns - 1; ph ^= 1u; }
        for (uint32_t t = 0; t < kLSpin && !mbar_try(smem_u32(&S.full[st]), ph ^ 1u); ++t) {}
    }
}

// ------------------------------------------------------------------ consumers
// what a chunk does not have in full: vectors beyond the task read as -inf, the row's ragged last vector loses the lanes
// beyond the vocabulary
template <int DT, int N>
__device__ __forceinline__ void mask_vecs(uint4* x, int vi, int nv, bool ragged, int keep) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
        if (vi + j * 32 >= nv) x[j] = neg_inf_vec<DT>();
        if (ragged && vi + j * 32 == nv - 1) mask_tail<DT>(x[j], keep);
    }
}
// Residuals of one vector pair: r' = max(0, e_p - rho e_q), rho as two floats, the large product first; as e_p <= 1, saturating
// to [0, 1] is the maximum with 0.  Their sum (the one that the finisher forms, sum_fixed).
template <int N>
__device__ __forceinline__ float resid_sum(const float* p, const float* q, float2 rho) {
    const float2 nh = make_float2(-rho.x, -rho.x);
    float2 z = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 t = __ffma2_rn(nh, make_float2(q[i], q[i + 1]), make_float2(p[i], p[i + 1]));
        const float2 r = make_float2(fma_sat(-rho.y, q[i], t.x), fma_sat(-rho.y, q[i + 1], t.y));
        z = i == 0 ? r : __fadd2_rn(z, r);
    }
    return z.x + z.y;
}
// bebop_tv: adds the residuals to *z and the e_q of the tokens with q <= p to *x.
template <int N>
__device__ __forceinline__ void resid_aux(const float* p, const float* q, float2 rho, float2* z, float2* x) {
    const float2 nh = make_float2(-rho.x, -rho.x), nl = make_float2(-rho.y, -rho.y);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 q2 = make_float2(q[i], q[i + 1]);
        const float2 d = __ffma2_rn(nl, q2, __ffma2_rn(nh, q2, make_float2(p[i], p[i + 1])));
        const float2 mk = make_float2(d.x >= 0.f ? 1.f : 0.f, d.y >= 0.f ? 1.f : 0.f);
        *z = __ffma2_rn(d, mk, *z);
        *x = __ffma2_rn(q2, mk, *x);
    }
}
// A warp's chunk of pass 1, from registers: its exponent, its sum and a bound of its sum of squares into the table.
template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_chunk1(FlowShared<F>& S, const uint4* x, float c, int par, int row, int at, int lane) {
    const QExp E = chunk_exponent(vecs_max<DT, F::LQV>(x), c);
    float sum;
    const int2 w = chunk_sum<DT, F::LQV, !TVM>(x, c, E.ef, &sum);
    // The lane's sum of e^2 is at most its sum of e, and at most that sum's square: the smaller, rounded up to 2^-15.
    const int sq = redux_add(__float_as_int(__fmaf_ru(__fmul_ru(sum, fminf(sum, 1.f)), 32768.f, kMagic)));
    if (lane == 0) S.part[par][row][at] = make_int4(w.x, w.y, E.e, sq);
}
// ... of pass 2: its mass (bebop_tv: and its part of S).
template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_chunk2(FlowShared<F>& S, const uint4* xp, const uint4* xq, float c, const float4& sc, int par, int at, int lane) {
    constexpr int VEC = Elem<DT>::VEC, H = F::LQV / 2;
    const float2 rho = make_float2(sc.z, sc.w);
    if (TVM) {
        float2 z = make_float2(0.f, 0.f), x = z;
#pragma unroll
        for (int i = 0; i < H; ++i) {
            float p[VEC], q[VEC];
            exp_vec<DT>(xp[i], c, sc.x, p);
            exp_vec<DT>(xq[i], c, sc.y, q);
            resid_aux<VEC>(p, q, rho, &z, &x);
        }
        const int2 w = warp_sum_words(z.x + z.y), v = warp_sum_words(x.x + x.y);
        if (lane == 0) { S.cm[par][at] = w; S.ca[par][at] = v; }
    } else {
        float v[H];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            float p[VEC], q[VEC];
            exp_vec<DT>(xp[i], c, sc.x, p);
            exp_vec<DT>(xq[i], c, sc.y, q);
            v[i] = resid_sum<VEC>(p, q, rho);
        }
        const int2 w = vector_sum_words<H, 0>(v);
        if (lane == 0) S.cm[par][at] = w;
    }
}

template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_consumer(const FlowArgs& a, FlowShared<F>& S, const unsigned char* ring, int warp, int lane) {
    constexpr int VEC = Elem<DT>::VEC;
    const int keep = a.r.V - (a.r.nvec - 1) * VEC;
#pragma unroll 1
    for (int st = -1, ph = 0;;) {
        if (++st == F::LNS) { st = 0; ph ^= 1; }
        const bool there = flow_wait_one(a, S, &S.full[st], (uint32_t)ph);
        const int4 d = S.task[st];
        // (one answer for the warp, as in flow_wait; voted here and not in front of the load: 1 per cent of a call)
        if (!__all_sync(0xffffffffu, there)) break;
        if ((d.x & 3) == 3) break;
        int j = warp - ((d.x >> 4) & 63);
        if (j < 0) j += F::LW;
        const int c0 = (d.x >> 16) + j, par = d.w & (F::LSL - 1), nv = d.y & 0xffff;
        const bool has = j < ((d.x >> 10) & 63);
        const int ragged = d.y >> 16;
        const float c = __int_as_float(d.z);
        if ((d.x & 3) == 0) {
            if (has) {
                const unsigned char* src = ring + (size_t)st * F::LSTAGE + (size_t)(j * F::LCV + lane) * 16;
                uint4 x[F::LQV];
#pragma unroll
                for (int i = 0; i < F::LQV; ++i) x[i] = *reinterpret_cast<const uint4*>(src + i * 512);
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.empty[st]);
                if ((j + 1) * F::LCV > nv - ragged) mask_vecs<DT, F::LQV>(x, j * F::LCV + lane, nv, ragged, keep);
                flow_chunk1<DT, TVM>(S, x, c, par, (d.x >> 2) & 1, c0, lane);
            } else { __syncwarp(); if (lane == 0) mbar_arrive(&S.empty[st]); }          // (every lane has read the description)
            if (lane == 0 && (d.x & 8)) mbar_arrive(&S.p1[par]);
        } else {
            const bool merged = flow_wait_one(a, S, &S.stat[par], ((uint32_t)d.w / F::LSL) & 1u);
            if (has) {
                const unsigned char* src = ring + (size_t)st * F::LSTAGE + (size_t)(j * (F::LCV / 2) + lane) * 16;
                constexpr int H = F::LQV / 2;
                uint4 xp[H], xq[H];
#pragma unroll
                for (int i = 0; i < H; ++i) { xp[i] = *reinterpret_cast<const uint4*>(src + i * 512); xq[i] = *reinterpret_cast<const uint4*>(src + F::LSTAGE / 2 + i * 512); }
                const float4 sc = S.scale[par];
                if (!__all_sync(0xffffffffu, merged)) break;
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.empty[st]);
                if ((j + 1) * (F::LCV / 2) > nv - ragged) {
                    mask_vecs<DT, H>(xp, j * (F::LCV / 2) + lane, nv, ragged, keep);
                    mask_vecs<DT, H>(xq, j * (F::LCV / 2) + lane, nv, ragged, keep);
                }
                flow_chunk2<DT, TVM>(S, xp, xq, c, sc, par, c0, lane);
            } else {
                if (!__all_sync(0xffffffffu, merged)) break;
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.empty[st]);
            }
            if (lane == 0 && (d.x & 8)) mbar_arrive(&S.p2[par]);
        }
        __syncwarp();
    }
}

// The consumers of the resident form: pass 1 of the unit that has arrived, pass 2 of the one `lag` before it, and its stage is free.
template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_consumer_res(const FlowArgs& a, FlowShared<F>& S, const unsigned char* ring, int warp, int lane) {
    constexpr int VEC = Elem<DT>::VEC, H = F::LQV / 2;
    const int keep = a.r.V - (a.r.nvec - 1) * VEC, lag = a.lag;
    int st = 0, st2 = 0, ph = 0;
    uint32_t end = 0xffffffffu;
#pragma unroll 1
    for (uint32_t u = 0;; ++u) {
        if (u < end) {
            const bool there = flow_wait_one(a, S, &S.full[st], (uint32_t)ph);
            const int4 d = S.task[st];
            if (!__all_sync(0xffffffffu, there)) return;
            if (d.x == 3) end = u;
            else {
                const int n1 = ((d.x >> 10) & 63) >> ((d.x >> 2) & 1), nv = d.y & 0xffff, par = u & (F::LSL - 1);      // chunks of a row
                int j = warp - ((d.x >> 4) & 63);
                if (j < 0) j += F::LW;
                if (j < ((d.x >> 10) & 63)) {
                    const int row = j >= n1 ? 1 : 0, jr = row ? j - n1 : j;
                    const unsigned char* src = ring + (size_t)st * a.pitch + (row ? a.pitch / 2 : 0) + (size_t)(jr * F::LCV + lane) * 16;
                    uint4 x[F::LQV];
#pragma unroll
                    for (int i = 0; i < F::LQV; ++i) x[i] = *reinterpret_cast<const uint4*>(src + i * 512);
                    if ((jr + 1) * F::LCV > nv - (d.y >> 16)) mask_vecs<DT, F::LQV>(x, jr * F::LCV + lane, nv, d.y >> 16, keep);
                    flow_chunk1<DT, TVM>(S, x, __int_as_float(d.z), par, row, jr, lane);
                }
                if (lane == 0) mbar_arrive(&S.p1[par]);
                if (++st == a.ns) { st = 0; ph ^= 1; }
            }
        }
        if (u >= (uint32_t)lag) {
            const uint32_t v = u - (uint32_t)lag;
            if (v >= end) return;
            const int par = v & (F::LSL - 1);
            const int4 d = S.task[st2];                      // (there since the unit's pass 1)
            const bool merged = flow_wait_one(a, S, &S.stat[par], (v / F::LSL) & 1u);
            int j = warp - ((d.x >> 16) & 63);
            if (j < 0) j += F::LW;
            const int nv = d.y & 0xffff;
            const bool has = j < ((d.x >> 22) & 63);
            if (!__all_sync(0xffffffffu, merged)) return;
            if (has) {
                const unsigned char* src = ring + (size_t)st2 * a.pitch + (size_t)(j * (F::LCV / 2) + lane) * 16;
                uint4 xp[H], xq[H];
#pragma unroll
                for (int i = 0; i < H; ++i) { xp[i] = *reinterpret_cast<const uint4*>(src + i * 512); xq[i] = *reinterpret_cast<const uint4*>(src + a.pitch / 2 + i * 512); }
                const float4 sc = S.scale[par];
                __syncwarp();
                if (lane == 0) mbar_arrive(&S.empty[st2]);
                if ((j + 1) * (F::LCV / 2) > nv - (d.y >> 16)) {
                    mask_vecs<DT, H>(xp, j * (F::LCV / 2) + lane, nv, d.y >> 16, keep);
                    mask_vecs<DT, H>(xq, j * (F::LCV / 2) + lane, nv, d.y >> 16, keep);
                }
                flow_chunk2<DT, TVM>(S, xp, xq, __int_as_float(d.z), sc, par, j, lane);
            } else { __syncwarp(); if (lane == 0) mbar_arrive(&S.empty[st2]); }
            if (lane == 0) mbar_arrive(&S.p2[par]);
            if (++st2 == a.ns) st2 = 0;
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ helper
// over the 16 lanes of a half warp, every lane gets the result (one fixed tree)
__device__ __forceinline__ int half_max(int v) {
    const bool low = (threadIdx.x & 16) == 0;
    const int a = redux_max(low ? v : INT_MIN), b = redux_max(low ? INT_MIN : v);
    return low ? a : b;
}
__device__ __forceinline__ double half_sum(double v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += shfl_xor_d(v, o);
    return v;
}

// The sums of pass 1, exchanged and merged.  Half a warp per row: lanes 0 to 15 the target row, 16 to 31 the draft row.
template <class F>
__device__ __forceinline__ void flow_exchange(const FlowArgs& a, FlowShared<F>& S, int rank, uint32_t first) {
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, C = a.C, row = lane >> 4, l = lane & 15;
    const int v0 = rank * a.sv, nv = max(min(a.sv, R.nvec - v0), 0), n1 = (nv + F::LCV - 1) / F::LCV;
#pragma unroll 1
    for (uint32_t u = first;; u += F::LNX) {
        if (!flow_wait(a, S, &S.ud[u % LUD], (u / LUD) & 1u)) return;
        const FlowUnit x = S.unit[u % LUD];
        const int par = u & (F::LSL - 1);
        if (x.b < 0) return;
        if (!flow_wait(a, S, &S.p1[par], (u / F::LSL) & 1u)) return;
        // ---- the CTA's sum of the row, sent to all CTAs of the cluster (a bonus row has an empty one beside it)
        const int n = row == 0 || x.pair() ? n1 : 0;
        const int4 none = make_int4(kNoSum0, kNoSum1, E_EMPTY, 0);
        const int4 v = l < n ? S.part[par][row][l] : none;
        int em = v.z;
        for (int q = l + 16; q < n; q += 16) em = max(em, S.part[par][row][q].z);
        em = half_max(em);
        const int bad = em == E_BAD;
        double s = 0.0, ub = 0.0;
        auto add = [&](const int4& v) {
            const double f = v.z > E_EMPTY && v.z != E_BAD ? pow2d(max(v.z - em, -500)) : 0.0;
            s = fma(2.0 * word_value(make_int2(v.x, v.y)), f, s);
            ub = fma(int_value((int)((unsigned)v.w - 32u * (unsigned)kMagicBits)), f * f, ub);
        };
        add(v);
        for (int q = l + 16; q < n; q += 16) add(S.part[par][row][q]);
        s = half_sum(s); ub = half_sum(ub);
        FlowRow m;
        int anybad = bad;
        m.e = em;
        if (C > 1) {
            if (l < C) {
                const uint32_t d = at_rank(&S.rrec[par][rank][row], l);
                st_remote(d, s); st_remote(d + 8, ub); st_remote(d + 16, em); st_remote(d + 20, bad);
                mbar_arrive_remote(at_rank(&S.rec[par], l));
            }
            __syncwarp();
        }
        if (a.expire) { if (lane == 0) flow_give_up(a, S); return; }          // test hook: this wait's bound has run out already
        if (C > 1) {
            if (!flow_wait<true>(a, S, &S.rec[par], (u / F::LSL) & 1u)) return;
            // ---- merged: the same bits in every CTA
            FlowRec r; r.s = 0.0; r.ub = 0.0; r.e = E_EMPTY; r.bad = 0;
            if (l < C) r = S.rrec[par][l][row];
            m.e = half_max(r.e);
            anybad = half_max(r.bad);
            const double f = r.e > E_EMPTY ? pow2d(max(r.e - m.e, -1000)) : 0.0;
            s = half_sum(r.s * f); ub = half_sum(r.ub * f * f);
        }
        m.st = (anybad || !(s == s)) ? ST_NONFINITE : m.e == E_EMPTY ? ST_EMPTY : 0;
        m.inv_s = !m.st && s > 0.0 ? 1.0 / s : 0.0; m.ub = ub * 3.0517578125e-05 * m.inv_s * m.inv_s; m.pad = 0.0;
        const double inv_q = __shfl_sync(0xffffffffu, m.inv_s, 16);
        const int eq = __shfl_sync(0xffffffffu, m.e, 16);
        if (!x.pair()) {
            // a bonus row has no pass 2: its chunks' masses are written now, before the consumers may use their places again
            const double inv_p = __shfl_sync(0xffffffffu, m.inv_s, 0);
            const int ep = __shfl_sync(0xffffffffu, m.e, 0);
            double t = 0.0;
            for (int q = lane; q < n1; q += 32) {
                const int4 w = S.part[par][0][q];
                const double v = w.z > E_EMPTY && w.z != E_BAD ? 2.0 * word_value(make_int2(w.x, w.y)) * pow2d(max(w.z - ep, -1000)) * inv_p : 0.0;
                a.mass[((int64_t)x.unit * C + rank) * (2 * a.nch) + q] = v;
                t += v;
            }
            t = warp_sum(t);
            if (lane == 0) a.smass[(int64_t)x.unit * C + rank] = t;
        }
        if (u >= F::LSL && !flow_wait(a, S, &S.pub[par], ((u - F::LSL) / F::LSL) & 1u)) return;
        if (lane == 0) {
            // (S_p / S_q; rows of equal sums have exactly 1)
            const double rh = !(m.inv_s > 0.0) ? 0.0 : inv_q == m.inv_s ? 1.0 : s * inv_q;
            const float h = (float)rh;
            S.scale[par] = make_float4((float)m.e, (float)eq, h, (float)(rh - (double)h));
            S.inv[par][0] = m.inv_s; S.inv[par][1] = inv_q;
        }
        if (rank == 0 && l == 0 && (row == 0 || x.pair())) a.rows[2 * (int64_t)x.unit + row] = m;
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.stat[par]);
        __syncwarp();
    }
}

// The masses of pass 2, written out, and the sequence's count; the last part of a sequence goes to the finisher.
template <bool TVM, class F>
__device__ __forceinline__ void flow_publish(const FlowArgs& a, FlowShared<F>& S, int rank) {
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, C = a.C;
    const int v0 = rank * a.sv, nv = max(min(a.sv, R.nvec - v0), 0), n2 = (nv + F::LCV / 2 - 1) / (F::LCV / 2);
    int parts = 0, b = 0, need = 0;
    flow_cleared();
    if (lane == 0) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");          // (the re-draw kernel reads what was cleared)
    auto deliver = [&](int b, int parts, int need) {
        __syncwarp();
        if (lane == 0) {
            __threadfence();
            if (atomicAdd(a.seqcnt + b, parts) == need - parts) {
                __threadfence();
                const int tail = S.mb_tail;
                bool room = false;
                for (uint32_t i = 0; i < kLSpin && !room; ++i) {
                    room = tail - *(volatile int*)&S.mb_head < LMB;
                    if (!room) { if (*(volatile int*)&S.abort) break; __nanosleep(100); }
                }
                if (!room) { atomicSub(a.seqcnt + b, parts); flow_give_up(a, S); }
                else {
                    S.mbox[tail % LMB] = b;
                    __threadfence_block();
                    *(volatile int*)&S.mb_tail = tail + 1;
                }
            }
        }
        __syncwarp();
    };
#pragma unroll 1
    for (uint32_t u = 0;; ++u) {
        if (!flow_wait(a, S, &S.ud[u % LUD], (u / LUD) & 1u)) break;
        const FlowUnit x = S.unit[u % LUD];
        const int par = u & (F::LSL - 1);
        if (x.b < 0) { if (parts) deliver(b, parts, need); break; }
        if (!flow_wait(a, S, &S.p2[par], (u / F::LSL) & 1u)) break;
        if (x.pair()) {
            const double ip = S.inv[par][0];
            double s = 0.0, sx = 0.0;
            for (int q = lane; q < n2; q += 32) {
                const double v = word_value(S.cm[par][q]) * ip;
                if (!TVM) a.mass[((int64_t)x.unit * C + rank) * (2 * a.nch) + q] = v;
                s += v;
                if (TVM) sx += word_value(S.ca[par][q]);
            }
            s = warp_sum(s);
            if (lane == 0) a.smass[(int64_t)x.unit * C + rank] = s;
            if (TVM) { sx = warp_sum(sx) * S.inv[par][1]; if (lane == 0) a.sauxp[(int64_t)x.unit * C + rank] = sx; }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.pub[par]);
        // the sequence's count takes the parts of a run of its units at once, with its last unit or this cluster's (the fence and
        // the atomic once per unit took as long as a short unit itself, and a cluster of one CTA sends itself nothing: 600
        // sequences of 8,000 bf16 logits, K = 7, 120.2 -> 101.4 us, 600 of 4,000 fp32, K = 8, 118.0 -> 89.7)
        ++parts; b = x.b; need = C * (TVM ? 1 : (x.kind >> 1) + 1);
        if (TVM || !x.pair()) { deliver(b, parts, need); parts = 0; }
        __syncwarp();
    }
    __syncwarp();
    if (lane == 0) { __threadfence_block(); *(volatile int*)&S.mb_done = 1; }
}

// ------------------------------------------------------------------ finisher
__device__ __forceinline__ FlowRow ld_flow_row(const FlowRow* p) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p)), w = __ldcg(reinterpret_cast<const double2*>(p) + 1);
    FlowRow x; x.inv_s = v.x; x.ub = v.y; x.e = __double2loint(w.x); x.st = __double2hiint(w.x); x.pad = 0.0;
    return x;
}
__device__ __forceinline__ FlowRow shfl_flow_row(const FlowRow& x, int src) {
    FlowRow y;
    y.inv_s = __shfl_sync(0xffffffffu, x.inv_s, src); y.ub = __shfl_sync(0xffffffffu, x.ub, src);
    y.e = __shfl_sync(0xffffffffu, x.e, src); y.st = __shfl_sync(0xffffffffu, x.st, src); y.pad = 0.0;
    return y;
}
__device__ __noinline__ void flow_finish_tv(const FlowArgs& a, int b) {
    const int lane = threadIdx.x & 31, C = a.C;
    const FlowRow rp = ld_flow_row(a.rows + 2 * (int64_t)b), rq = ld_flow_row(a.rows + 2 * (int64_t)b + 1);
    const int st = tau_ok(tau_of(a.r, b)) ? (rp.st | rq.st) : ST_BAD_TEMP;
    double z = lane < C ? __ldcg(a.smass + (int64_t)b * C + lane) : 0.0, x = lane < C ? __ldcg(a.sauxp + (int64_t)b * C + lane) : 0.0;
    z = warp_sum(z); x = warp_sum(x);
    if (lane == 0) {
        a.o.tv[b] = st ? 0.f : (float)fmin(fmax(z, 0.0), 1.0);
        if (a.s_aux) a.s_aux[b] = st ? 0.f : (float)x;
        if (a.o.row_status) a.o.row_status[b] = st;
    }
}
// One warp; what it reads was published before the sequence's count reached its last value.
template <int DT, class F>
__device__ __noinline__ void flow_finish(const FlowArgs& a, int b) {
    constexpr int VEC = Elem<DT>::VEC;
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, K = R.K, V = R.V, C = a.C, L = len_of(R, b);
    const float tau = tau_of(R, b), c = temp_scale(tau).hi;
    int seq_st = tau_ok(tau) ? 0 : ST_BAD_TEMP;
    const int64_t unit0 = (int64_t)b * (K + 1);
    // ---- lane k owns draft position k; what does not depend on each other is asked for together
    const bool active = lane < L;
    const int tk = active ? a.draft_tokens[(int64_t)b * K + lane] : 0;
    const float u = active ? a.u_accept[(int64_t)b * K + lane] : 0.f;
    const float uf = a.u_final[b];
    const bool tok_ok = tk >= 0 && tk < V;
    float zpx = 0.f, zqx = 0.f;
    if (active && tok_ok) { zpx = load_one<DT>(row_ptr(R, b, lane), tk); zqx = load_one<DT>(row_ptr(R, b, K + 1 + lane), tk); }
    FlowRow sp, sq;
    sp.inv_s = 0.0; sp.ub = 0.0; sp.e = E_EMPTY; sp.st = 0; sp.pad = 0.0; sq = sp;
    if (active) { sp = ld_flow_row(a.rows + 2 * (unit0 + lane)); sq = ld_flow_row(a.rows + 2 * (unit0 + lane) + 1); }
    const FlowRow sb = ld_flow_row(a.rows + 2 * (unit0 + L));
    double tv = 0.0;
    if (active) for (int r = 0; r < C; ++r) tv += __ldcg(a.smass + (unit0 + lane) * C + r);
    if (!seq_st && __ballot_sync(0xffffffffu, active && !tok_ok)) seq_st = ST_BAD_TOKEN;
    // the first bad row pair decides the status; rows after it do not count
    const int rs = active ? (sp.st | sq.st) : 0;
    const unsigned badrows = __ballot_sync(0xffffffffu, rs != 0);
    const int first_bad = badrows ? __ffs(badrows) - 1 : 32;
    const int rs_first = __shfl_sync(0xffffffffu, rs, first_bad & 31);
    if (!seq_st && badrows) seq_st = rs_first;
    double px = 0.0, qx = 0.0;
    bool acc = false;
    if (active && !(seq_st & ST_FATAL) && lane < first_bad) {
        const double cd = (double)c;
        px = exp2((double)zpx * cd - (double)sp.e) * sp.inv_s;
        qx = exp2((double)zqx * cd - (double)sq.e) * sq.inv_s;
        acc = (double)u * qx < px;
    }
    const unsigned rej = __ballot_sync(0xffffffffu, active && !acc);
    const int n = rej ? __ffs(rej) - 1 : L;
    if (!(seq_st & ST_FATAL) && n == L) seq_st |= sb.st;              // bonus row, counted only now
    const bool fatal = (seq_st & ST_FATAL) != 0;
    const int nn = fatal ? 0 : n;
    for (int q = lane; q <= K; q += 32)
        if (fatal || q != nn) a.o.out_tokens[(int64_t)b * (K + 1) + q] = q < nn ? tk : -1;          // (q < nn <= 32: q == lane)
    if (lane < K) {
        const bool zero = fatal || lane >= L;
        if (a.o.p_draft) a.o.p_draft[(int64_t)b * K + lane] = zero ? 0.f : (float)px;
        if (a.o.q_draft) a.o.q_draft[(int64_t)b * K + lane] = zero ? 0.f : (float)qx;
        if (a.o.tv) a.o.tv[(int64_t)b * K + lane] = zero ? 0.f : (float)fmin(fmax(tv, 0.0), 1.0);
    }
    if (lane == 0) {
        a.o.accept_len[b] = nn;
        if (a.o.row_status) a.o.row_status[b] = seq_st;
    }
    if (fatal) { if (lane == 0) draw_decided(a.fb_count); return; }
    // ---- the draw: position nn (row pair), or the bonus row when every draft was accepted
    const bool pair = nn < L;
    const FlowRow rp = pair ? shfl_flow_row(sp, nn) : sb;
    FlowRow rq = shfl_flow_row(sq, pair ? nn : 0);
    if (!pair) { rq.inv_s = 0.0; rq.ub = 0.0; rq.e = 0; }
    const double bound = draw_bound(rp.ub + rq.ub, (double)a.kappa);
    const int64_t du = unit0 + nn;
    double base, total;
    const double m = lane < C ? __ldcg(a.smass + du * C + lane) : 0.0;
    owner_lane(m, 0.0, -1.0, &base, &total);
    const double Tt = (double)uf * total;
    int y = -1, cert = 0;
    double tot;
    const int own = Tt > 0.0 ? owner_lane(m, 0.0, Tt, &base, &tot) : -1;
    if (own >= 0) {
        const int v0 = own * a.sv, nv = max(min(a.sv, R.nvec - v0), 0), cv = pair ? F::LCV / 2 : F::LCV, nc = (nv + cv - 1) / cv;
        int ch = -1;
        double at = base;
        for (int g = 0; g < nc && ch < 0; g += 32) {
            double b0;
            const int ow = owner_lane(g + lane < nc ? __ldcg(a.mass + (du * C + own) * (2 * a.nch) + g + lane) : 0.0, at, Tt, &b0, &tot);
            if (ow >= 0) { ch = g + ow; at = b0; } else at = tot;
        }
        if (ch >= 0) {
            const double r = rp.inv_s > 0.0 ? rq.inv_s / rp.inv_s : 0.0;
            const float2 rho = make_float2((float)r, (float)(r - (double)(float)r));
            const char* prow = row_ptr(R, b, nn) + (int64_t)v0 * 16;
            const char* qrow = pair ? row_ptr(R, b, K + 1 + nn) + (int64_t)v0 * 16 : prow;
            const int vend = min(nv, (ch + 1) * cv);
#pragma unroll 1
            for (int j = 0; j < cv / 32; ++j) {
                const int vi = ch * cv + j * 32 + lane, left = V - (v0 + vi) * VEC;
                uint4 xp = neg_inf_vec<DT>(), xq = xp;
                if (vi < vend) { xp = ldg16(prow + (int64_t)vi * 16); if (pair) xq = ldg16(qrow + (int64_t)vi * 16); }
                if (vi < vend && left < VEC) { mask_tail<DT>(xp, left); mask_tail<DT>(xq, left); }
                float e[VEC], q[VEC];
                exp_vec<DT>(xp, c, (float)rp.e, e);
                exp_vec<DT>(xq, c, (float)rq.e, q);
                if (pair)
#pragma unroll
                    for (int i = 0; i < VEC; i += 2) {
                        const float2 t = __ffma2_rn(make_float2(-rho.x, -rho.x), make_float2(q[i], q[i + 1]), make_float2(e[i], e[i + 1]));
                        e[i] = fma_sat(-rho.y, q[i], t.x); e[i + 1] = fma_sat(-rho.y, q[i + 1], t.y);
                    }
                const double dv = (double)sum_fixed<VEC>(e) * rp.inv_s;
                double incl = dv;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
                const double lo = at + (incl - dv), hi = at + incl;
                if (y < 0 && lo < Tt && Tt <= hi) {
                    double Cw = lo;
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        const double r1 = (double)e[i] * rp.inv_s, Cn = Cw + r1;
                        if (y < 0 && r1 > 0.0 && Cn >= Tt) { y = (v0 + vi) * VEC + i; cert = (Tt - Cw > bound) && (Cn - Tt >= bound); }
                        Cw = Cn;
                    }
                }
                at += __shfl_sync(0xffffffffu, incl, 31);
            }
        }
    }
    const unsigned found = __ballot_sync(0xffffffffu, y >= 0);
    const bool ok = __popc(found) == 1 && __shfl_sync(0xffffffffu, cert, (__ffs(found) - 1) & 31);
    if (ok) {
        if (y >= 0) { a.o.out_tokens[(int64_t)b * (K + 1) + nn] = y; draw_decided(a.fb_count); }
    } else if (lane == 0) st_fb(a.fb_list + draw_listed(a.fb_count), b, 2 * nn + (pair ? 1 : 0), rp.e, pair ? rq.e : 0);
    __syncwarp();
}

// One warp completes sequences while the stream goes on; the consumers help with what has been left when they are through (a
// sequence takes a warp some ten microseconds, so that calls of many short rows leave a good part of them: 600 sequences of 8,000
// bf16 logits, K = 7, 96.6 -> 93.2 us, 192 of 32,000, K = 7 ragged, 69.2 -> 61.6, 1,000 of 8,000 fp32 107.5 -> 92.7).
template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_finisher(const FlowArgs& a, FlowShared<F>& S) {
    const int lane = threadIdx.x & 31;
    for (;;) {
        int b = -1, done = 0;
        if (lane == 0) {
            done = *(volatile int*)&S.mb_done;                      // read before the tail: entries come first
            __threadfence_block();
            const int head = *(volatile int*)&S.mb_head;
            if (head != *(volatile int*)&S.mb_tail) {
                // (an entry is read before it is taken: once taken, its place may be written again)
                __threadfence();
                b = *(volatile int*)&S.mbox[head % LMB];
                done = 0;
                if (atomicCAS(&S.mb_head, head, head + 1) != head) b = -2;
            }
        }
        b = __shfl_sync(0xffffffffu, b, 0); done = __shfl_sync(0xffffffffu, done, 0);
        if (b >= 0) {
            __threadfence();                                        // (the other lanes read behind lane 0's look)
            if (TVM) flow_finish_tv(a, b); else flow_finish<DT, F>(a, b);
            __syncwarp();
            continue;
        }
        if (done) break;
        if (b == -1) __nanosleep(40);
    }
}

// A CTA that gave up: the sequences that nobody has completed and nobody will say so in their outputs.  The count decides, in the one
// access that marks it: whoever delivers a last part afterwards finds the mark and completes nothing.
template <bool TVM, class F>
__device__ __noinline__ void flow_failed(const FlowArgs& a) {
    const RowArgs& R = a.r;
    const int K = R.K;
    for (int b = threadIdx.x; b < R.B; b += F::LT) {
        const int need = a.C * (TVM ? 1 : len_of(R, b) + 1);
        if (ld_acquire(a.seqcnt + b) >= need) continue;
        const int old = atomicOr(a.seqcnt + b, kFailed);         // (added, two marks would overflow into a count that looks open)
        if ((old & kFailed) || old >= need) continue;
        if (TVM) { a.o.tv[b] = 0.f; if (a.s_aux) a.s_aux[b] = 0.f; }
        else {
            a.o.accept_len[b] = 0;
            for (int q = 0; q <= K; ++q) a.o.out_tokens[(int64_t)b * (K + 1) + q] = -1;
            for (int k = 0; k < K; ++k) {
                const int64_t i = (int64_t)b * K + k;
                if (a.o.tv) a.o.tv[i] = 0.f;
                if (a.o.p_draft) a.o.p_draft[i] = 0.f;
                if (a.o.q_draft) a.o.q_draft[i] = 0.f;
            }
            draw_decided(a.fb_count);
        }
        if (a.o.row_status) a.o.row_status[b] = ST_WAIT;
    }
}

template <int DT, bool TVM, class F>
__device__ __forceinline__ void flow_body(const FlowArgs& a, unsigned char* smem) {
    FlowShared<F>& S = *reinterpret_cast<FlowShared<F>*>(smem + F::LRING);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = a.C > 1 ? (int)cluster_rank() : 0, g = (int)blockIdx.x / a.C;
    if (tid == 0) {
        for (int i = 0; i < F::LNS; ++i) { mbar_init(&S.full[i], 1); mbar_init(&S.empty[i], F::LW); }
        for (int i = 0; i < LUD; ++i) mbar_init(&S.ud[i], 1);
        for (int i = 0; i < F::LSL; ++i) { mbar_init(&S.p1[i], F::LW); mbar_init(&S.p2[i], F::LW); mbar_init(&S.rec[i], 2 * a.C); mbar_init(&S.stat[i], 1); mbar_init(&S.pub[i], 1); }
        S.mb_tail = 0; S.mb_head = 0; S.mb_done = 0; S.abort = 0;
        S.start_b = a.r.B; S.start_k = 0; S.start_w = 0; S.end_w = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    flow_share<TVM>(a, S, g);
    __syncthreads();
    if (a.C > 1) cluster_sync();                            // every CTA of the cluster has its barriers
    if (warp < F::LW) {
        if constexpr (F::LRES) flow_consumer_res<DT, TVM>(a, S, smem, warp, lane); else flow_consumer<DT, TVM>(a, S, smem, warp, lane);
        flow_finisher<DT, TVM>(a, S);
    } else if (warp == F::W_FPROD) {
        if (lane == 0) { if constexpr (F::LRES) flow_producer_res<DT, TVM>(a, S, smem, rank); else flow_producer<DT, TVM>(a, S, smem, rank); }
        __syncwarp();
    } else if (warp == F::W_PUB) flow_publish<TVM>(a, S, rank);
    else if (warp == F::W_FIN) flow_finisher<DT, TVM>(a, S);
    else flow_exchange(a, S, rank, (uint32_t)(warp - F::W_EXCH));
    __syncthreads();
    if (a.C > 1) cluster_sync();                            // nothing is sent to a CTA that has left
    if (*(volatile int*)&S.abort) flow_failed<TVM, F>(a);
}

// ------------------------------------------------------------------ host side
template <class F> constexpr size_t flow_smem() { return F::LRING + sizeof(FlowShared<F>); }

// The smallest share, in rows, that G clusters of at most that many take all units with (a row pair is not cut), for calls of a few
// rows per cluster, where even shares leave some clusters a row more (48 sequences of 151,936, K = 3, 65.1 -> 61.0 us, 30 of 200,000,
// K = 2, 50.3 -> 47.7).  From five rows on the even shares stay (0): they leave some clusters a row less, and are done
// sooner (64 of 151,936 71.9 against 77.9 us, 256 of them 177.9 against 179.6).
inline int flow_share_of(const RowArgs& a, bool tv_only, int G) {
    const int w = tv_only ? 2 : 2 * a.K + 1, total = a.B * w;
    if (total >= 5 * G) return 0;
    for (int share = (total + G - 1) / G < 2 ? 2 : (total + G - 1) / G;; ++share) {
        int at = 0, r = 0;
        for (int g = 0; g < G && at < total; ++g) flow_next(at, r, share, share % w, w);
        if (at >= total) return share;
    }
}
// Multiprocessors of the device (asked once per device).
inline int flow_sms() {
    static int cached[64] = {0};
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 148; }
    if (!cached[dev]) {
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { cudaGetLastError(); return 148; }
        cached[dev] = n;
    }
    return cached[dev];
}
// Clusters of so many CTAs for a call.  Two units of every cluster have to stay in L2, and the tables hold 20,480 vectors of a slice:
// one CTA up to 10,240 vectors per row, two up to 40,960, and so on.  Above that the least work of the busiest cluster decides: the
// rows of its share, each a slice and what a unit costs beside it, in vectors -- exchanges of two CTAs hide under 130, of four and
// eight they cost 1,300 and 800 where few units come between (us per call on a B200 with one, two, four, eight CTAs, bf16; fitted to 110
// such calls: bebop_tv of 300 row pairs of 65,536 40, 36, 43, 59; 100 of 100,000 -, 27, 29, 31; 100 of 262,144 -, 50, 49, 46;
// K = 3: 200 sequences of 65,536 77, 85, 92, 136; 24 of 151,936 -, 37, 39, 41; 12 of 151,936 -, 35, 32, 30; 4 of 151,936, K = 8, -,
// 33, 27.5, 27.6; 512 of 262,144 -, 537, 546, -).
inline int flow_cluster(const RowArgs& a, bool tv_only) {
    constexpr int kUnit[kFlowMaxCluster + 1] = {0, 0, 130, 0, 1300, 0, 0, 0, 800};
    int C = 1, best = 0;
    while (C < kFlowMaxCluster && a.nvec > (C == 1 ? 10240 : 20480 * C)) C *= 2;
    const double rows = (double)a.B * (tv_only ? 2 : 2 * a.K + 1);
    double least = 0.0;
    for (; C <= kFlowMaxCluster; C *= 2) {
        const int G = flow_sms() / C > 0 ? flow_sms() / C : 1, share = flow_share_of(a, tv_only, G);
        const double t = (share ? (double)share : rows / G) * ((double)a.nvec / C + kUnit[C]);
        if (!best || t < least) { best = C; least = t; }
        if (a.nvec <= 4 * 256 * C) break;
    }
    return best;
}
inline bool flow_resident_rows(const RowArgs& a, int C) { return C == 1 && a.nvec <= kResidentVecs; }
// Large chunks for long slices (row pairs of 151,936 over two CTAs 152.7 against 164.7 us for 768 of them; 192 sequences of 32,000,
// K = 7, over one CTA 79.7 against 70.0; 24 of 151,936 over four 45.0 against 42.3; 500 of 50,000 over one 155 against 133; 500 of 90,000 over
// two, slices of 5,600 vectors, 235 against 208, 200 of 100,000, K = 8, slices of 6,300, 226 against 231).
inline bool flow_long(const RowArgs& a, bool tv_only, int C) { return a.nvec > (tv_only ? 4000 : C == 1 ? 7500 : 6000) * C; }
template <class F, auto kernel> bool flow_ready() {
    static bool done[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (dev >= 0 && dev < 64 && done[dev]) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)flow_smem<F>()) != cudaSuccess) { cudaGetLastError(); return false; }
    if (dev >= 0 && dev < 64) done[dev] = true;
    return true;
}
// how many clusters of C CTAs the device holds at a time (asked once per device; 0: not known)
template <class F, auto kernel> int flow_resident(int C) {
    static int cached[64][kFlowMaxCluster + 1] = {{0}};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 0; }
    int& n = cached[dev][C];
    if (n) return n > 0 ? n : 0;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C); cfg.blockDim = dim3(F::LT); cfg.dynamicSmemBytes = flow_smem<F>();
    cfg.attrs = attr; cfg.numAttrs = 1;
    int got = 0;
    if (!flow_ready<F, kernel>() || cudaOccupancyMaxActiveClusters(&got, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); got = 0; }
    n = got > 0 ? got : -1;
    return got > 0 ? got : 0;
}
struct FlowCall {
    const RowArgs& a; const Plan& p;
    const int32_t* draft_tokens; const float* u_accept; const float* u_final;
    VerifyOut o; char* ws; cudaStream_t stream; bool tv_only; float* s_aux;
};
// One call with clusters of C CTAs through `kernel`; *launched stays false where the shape, the workspace or the device
// has no room for it.
template <class F, auto kernel> cudaError_t flow_launch(const FlowCall& x, int C, bool* launched) {
    static_assert(flow_smem<F>() <= 232448, "shared memory of a CTA");
    *launched = false;
    const RowArgs& a = x.a;
    const FlowPlan f = make_flow_plan(a.B, a.K, a.nvec, x.tv_only ? 1 : a.K + 1, C, F::LCV);
    static_assert(2 * sizeof(FlowRow) <= 80, "rows in the plan");
    if (a.K > BEBOP_MAX_K_INT || f.nch > F::MAXCH || (long long)a.B * (2 * a.K + 1) >= 0x7fffffffLL || f.total > x.p.total - x.p.off_pipe) return cudaSuccess;
    const int G = flow_resident<F, kernel>(C);
    if (G < 1 || !flow_ready<F, kernel>()) return cudaSuccess;
    char* w = x.ws + x.p.off_pipe;
    FlowArgs fa;
    fa.r = a; fa.draft_tokens = x.draft_tokens; fa.u_accept = x.u_accept; fa.u_final = x.u_final; fa.o = x.o; fa.s_aux = x.tv_only ? x.s_aux : nullptr;
    fa.C = C; fa.nch = f.nch; fa.sv = f.sv;
    // small chunks: an exchange may take longer than a unit's work, so more units go between (600 sequences of 8,000 bf16 logits, K = 7:
    // one 101.4, two 98.7, three 96.7 us; 96 of 65,536, K = 1, over two CTAs 38.1, 35.6, 35.6; 12 of 151,936 over eight 30.7, 29.6, 29.5);
    // longer slices have no use for it, and L2 has to hold them
    fa.lag = F::LSL > 3 ? (a.nvec <= 2560 ? 3 : 2) : 1;
    fa.ns = 0; fa.pitch = 0;
    if (F::LRES) {
        fa.pitch = 2 * ((min(f.sv, a.nvec) * 16 + 127) & ~127);
        fa.ns = min(F::LNS, F::LRING / fa.pitch);
        fa.lag = min(3, fa.ns - 2);
    }
    const long long units = (long long)a.B * (x.tv_only ? 1 : a.K + 1);
    fa.G = (int)(units < G ? units : G);
    fa.share = x.tv_only || !a.draft_len ? flow_share_of(a, x.tv_only, fa.G) : -1;
    const int expire = take_expire_wait();
    fa.expire = expire == 2 ? 1 : 0;
    fa.kappa = draw_kappa();
    fa.wait_failed = reinterpret_cast<int*>(w) + 1;
    fa.fb_count = reinterpret_cast<unsigned long long*>(w + kFbCountOffset);
    fa.fb_list = reinterpret_cast<FbRec*>(w + f.off_fbrec);
    fa.seqcnt = reinterpret_cast<int*>(w + f.off_seqcnt);
    fa.rows = reinterpret_cast<FlowRow*>(w + f.off_rows);
    fa.smass = reinterpret_cast<double*>(w + f.off_smass);
    fa.sauxp = reinterpret_cast<double*>(w + f.off_saux);
    fa.mass = reinterpret_cast<double*>(w + f.off_mass);
    cudaError_t e = clear_launch(w, f.zero_bytes, x.stream);
    if (e != cudaSuccess) return e;
    if (g_ev_start) cudaEventRecord(g_ev_start, x.stream);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = C; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(fa.G * C)); cfg.blockDim = dim3(F::LT); cfg.dynamicSmemBytes = flow_smem<F>(); cfg.stream = x.stream;
    cfg.attrs = attr; cfg.numAttrs = C > 1 ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, kernel, fa);
    if (g_ev_stop) cudaEventRecord(g_ev_stop, x.stream);
    if (e != cudaSuccess) { cudaGetLastError(); return cudaSuccess; }        // (no room for such a cluster: the caller takes another kernel)
    *launched = true;
    if (x.tv_only) return cudaSuccess;
    // the fp64 re-draw of the listed sequences, on the same workspace head and list
    PipePlan wp = make_pipe_plan(a.B, a.K, a.nvec, a.dt);
    wp.off_xsdone = f.off_xsdone; wp.off_xdone = f.off_xdone; wp.off_xsum = f.off_xsum; wp.off_xmass = f.off_xmass;
    return redraw_launch(a, x.u_final, x.o, fa.fb_count, fa.fb_list, a.B, fa.wait_failed, w, wp, x.stream, expire == 1);
}

}  // namespace

}  // namespace bebop
