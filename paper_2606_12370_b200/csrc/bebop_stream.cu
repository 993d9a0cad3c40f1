// Streaming kernel: bebop_verify and bebop_tv with every logit row read from memory once and exponentiated once, in ONE
// launch (clearing of the workspace, sweep, accept scan, draw and fp64 re-draw).
//
// A row (pair) is cut into T slices of at most 2048 16-byte vectors; a task is one slice of a row pair (target row k,
// draft row k of a sequence: a "unit") or two slices of a sequence's bonus row.  Tasks are dealt round robin over a grid
// that is resident as a whole (one CTA per SM), so the T slices of a unit are in the hands of T CTAs at about the
// same time.  Sixteen consumer warps own a chunk of 128 vectors each.  Per task they
//   pass 1  take the chunk of either row from shared memory (bulk copies, a ring of one-row stages), form
//           e = 2^(x c - E) around an integer reference exponent E per chunk, and park the e -- in TENSOR MEMORY (this path has
//           no contraction, so the 256 KB of TMEM per SM are free to serve as a store) and, as a third task's place, in shared
//           memory; their sums go to a stats warp, which stores the slice's softmax partial (E, sum e) as a record in
//           global memory, finds the T records of the unit, merges them -- exact power-of-two scalings, one fixed
//           order, so every CTA gets the same bits -- and so knows both normalisers S_p, S_q;
//   pass 2  take the e back, when the normalisers are known, and form r' = max(0, e_p - rho e_q), rho = S_p / S_q as two
//           floats: the residual p - q up to the factor 1 / S_p, which is applied once per unit, in double.
// Pass 2 of a task runs in quarters between the halves of pass 1 of later tasks: the exponential unit works on one warp's
// chunk while another's residuals are formed (the two passes one after the other left it idle a third of the time).
// Finisher warps complete sequences: accept scan (Algorithm 3) as soon as the rows' normalisers are there, then, when the
// masses are, the chunk that owns the target u Z of the inverse CDF and the token in it, kept if the crossing clears the
// error bound; else the sequence is listed, and the consumer warps, when they have run out of tasks, evaluate the
// listed sequences' draw rows again in double.
//
// What CTAs pass to each other are words that are valid by themselves once non-zero (the memory is cleared by the kernel,
// before the grid meets once), written and read by relaxed accesses: no fence on the streaming path.  Every wait is
// bounded; one that gives up sets the wait flag and lets the CTA run out (status bit 32 of every row).  No cluster.
// Tasks wait only for tasks of earlier rounds of the deal (a CTA's task n waits for the units of its task n - NSLOT),
// so nothing can deadlock.
#include <cooperative_groups.h>

#include "bebop_chunk.cuh"

namespace bebop {

namespace {

constexpr int CW = kStreamWarps;              // consumer warps = chunks of a slice
constexpr int CV = kStreamChunkVecs;          // vectors per chunk and row: four per lane
constexpr int CH = CW;
constexpr int SV = kStreamSliceVecs;          // vectors per slice, at most
static_assert(CW == 12 && CH % 4 == 0 && CV == 128 && SV == CH * CV, "slice size, chunks, TMEM columns per warp");
constexpr int NSTG = 6;                       // stages of the ring of logits: one row of a slice each
constexpr int STAGE = SV * 16;
constexpr int RING = NSTG * STAGE;
#ifndef BS_NSTAT
#define BS_NSTAT 2
#endif
#ifndef BS_NF
#define BS_NF 1
#endif
#ifndef S_FULL
#define S_FULL 32
#endif
#ifndef S_STAT
#define S_STAT 32
#endif
#ifndef S_PD
#define S_PD 64
#endif
#ifndef S_EMPTY
#define S_EMPTY 64
#endif
#ifndef S_LOOK
#define S_LOOK 150
#endif
constexpr int NSTAT = BS_NSTAT;               // stats warps
constexpr int NFIN = BS_NF;                   // finisher warps
constexpr int R8 = 8;                         // ring of the barriers of a task
constexpr int RT = 16;                        // ring of the descriptions: the end's are written up to NSTAT ahead of the last task's
constexpr int W_PROD = CW, W_STAT0 = CW + 1, W_FIN0 = W_STAT0 + NSTAT;
constexpr int ST_THREADS = (W_FIN0 + NFIN) * 32;
constexpr int TCOLS = 512;                    // TMEM columns of a CTA
constexpr int kPair = 0, kBonus = 1, kStop = 2;
constexpr uint32_t kWaitSpin = 1u << 23;
constexpr int XV = 64;                        // vectors of an item of the re-draw: two per lane

template <int DT> struct Dims {
    static constexpr int VEC = Elem<DT>::VEC;
    static constexpr int TCOL = 2 * 4 * VEC;                   // TMEM columns of a task: per vector VEC of the target row, VEC of the draft row
    static constexpr int WCOL = 160;                           // columns of a warp: three warps share a quarter of the lanes
    // Tasks whose exponentials wait at a time.  bf16: two and a half of them in the warp's columns, the last two vectors of
    // every third task in shared memory.
    static constexpr int NSLOT = DT == 1 ? 3 : 4;
    static constexpr int MWARP = NSLOT * TCOL > WCOL ? 2 * 32 * 2 * VEC * 4 : 0;      // bytes of a warp's part in shared memory
    static constexpr int DATA = RING + CW * MWARP;
    static_assert((NSLOT - 1) * TCOL + TCOL / (MWARP ? 2 : 1) <= WCOL && 3 * WCOL <= TCOLS, "columns");
    static_assert(NSLOT == 3 || NSLOT == 4, "rings");
};

// One task: slice s of target row k and draft row k of a sequence, or (bonus) two slices, s and s + 1, of its bonus
// row, the second in the draft row's place, so that the bonus row costs per byte what the row pairs cost.
struct __align__(16) Task {
    float c;                             // log2(e) / tau
    int meta;                            // kind (2 bits), vectors of the first and the second row (12 each), the row's last vector is ragged
    int us, unit;                        // unit * T + s
};
__device__ __forceinline__ int t_kind(int m) { return m & 3; }
__device__ __forceinline__ int t_nv(int m) { return (m >> 2) & 0xfff; }
__device__ __forceinline__ int t_nv2(int m) { return (m >> 14) & 0xfff; }
__device__ __forceinline__ bool t_tail(int m) { return (m >> 26) & 1; }
// Softmax partial of one slice of one row; each 8-byte word is valid by itself once non-zero.  `flags`: bit 0 says
// that the slice holds a NaN or +inf; the other bits are those of a float u that bounds the slice's sum of e^2
// (around the slice's exponent) from above: e <= 1, so a chunk's is at most its sum of e.
struct __align__(16) Rec { double s; int ecode; int flags; };
// (an exponent is stored as e + 2^24, far from zero and from the ends of the integers; 1: the slice holds nothing but -inf)
constexpr int kCodeBias = 1 << 24, kCodeEmpty = 1;
__device__ __forceinline__ int rec_e(const Rec& r) { return r.ecode == kCodeEmpty ? E_EMPTY : r.ecode - kCodeBias; }
__device__ __forceinline__ int rec_code(int e) { return e > E_EMPTY ? e + kCodeBias : kCodeEmpty; }
__device__ __forceinline__ float rec_ub(const Rec& r) { return __int_as_float(r.flags & ~1); }
__device__ __forceinline__ Rec no_rec() { Rec r; r.s = 0.0; r.ecode = kCodeEmpty; r.flags = 0; return r; }
struct __align__(16) Row { double inv_s; int e; int st; };            // a merged row: 1/S, exponent, status bits (| kRowValid)

struct StreamArgs {
    RowArgs r;
    const int32_t* draft_tokens;
    const float* u_accept;
    const float* u_final;
    VerifyOut o;
    float* s_aux;
    int ups;                 // units per sequence: K + 1 (row pairs, bonus row), or 1 for bebop_tv
    int tps;                 // tasks per sequence
    int T, slice_vecs, total, nx;  // nx: items of the re-draw per sequence
    int expire;              // test hook: 1 the re-draw's wait for the list, 2 the stats warps' wait gives up at once
    float kappa;
    char* zero; unsigned zero16;   // what the kernel clears before anything else: 16-byte words
    int* wait_failed;
    unsigned* xticket;
    unsigned long long* fb_count;
    FbRec* fb_list;
    Rec* rec;                // [units][T][2]
    float* cm;               // [units][T][CH] residual mass per chunk (bonus row: sum of e around the slice's exponent)
    float* ca;               // [units][T][CH] bebop_tv: sum of q over the tokens with q <= p
    Row* rows;               // [units][2] the merged rows of a row pair
    double2* xsum;           // [B][nx] re-draw: sums of exponentials per item, by place in the list
    double* xmass;           // [B][nx] ... and residual masses
};

struct Shared {
    unsigned long long full[NSTG], empty[NSTG];
    unsigned long long pdone[R8];            // the consumers' sums of the task are there
    unsigned long long stats[R8];            // the task's rho is there
    unsigned long long fbcount;              // copy of the list's counters for this CTA's warps
    Task task[RT];
    double tab[64];                          // 2^(j/64)
    uint32_t tmem_base;
    int abort, failed;
};
// Per task: first the chunks' sums (fixed point, two words) and exponents, target row and draft row; then, in place of
// the target row's, rho (two floats) and the factors that bring the chunk's residuals to the rows' exponents.
struct __align__(16) Slot { union { int4 part[2][CH]; float4 rho[CH]; }; };
template <int DT> struct SharedD : Shared { Slot slot[Dims<DT>::NSLOT]; };
static_assert(sizeof(SharedD<1>) + Dims<1>::DATA <= 232448, "shared memory of a CTA");

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ void mbar_arrive(uint32_t addr) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(addr) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) { mbar_arrive(smem_u32(b)); }
// Bounded; gives up at once when the CTA has already given up somewhere.  Sleeps between looks: a warp that spins takes
// issue slots from the warp it waits for (try_wait itself returns within 30 cycles, whatever its time hint).
template <int NS>
__device__ __forceinline__ bool mbar_wait(Shared& S, uint32_t addr, uint32_t parity) {
    if (mbar_try(addr, parity)) return true;
    for (uint32_t i = 0; i < kWaitSpin; ++i) {
        __nanosleep(NS);
        if (mbar_try(addr, parity)) return true;
        if (*(volatile int*)&S.abort) return false;
    }
    return false;
}
__device__ __forceinline__ uint4 lds16(uint32_t p) {
    uint4 v; asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(p) : "memory"); return v;
}
__device__ __forceinline__ float4 lds16f(uint32_t p) {
    float4 v; asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(p) : "memory"); return v;
}
__device__ __forceinline__ void sts16(uint32_t p, const float* e) {
    asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" :: "r"(p), "f"(e[0]), "f"(e[1]), "f"(e[2]), "f"(e[3]) : "memory");
}
__device__ __forceinline__ float set_ge0(float d) {          // 1.0 where d >= 0, else 0.0
    float m; asm("set.ge.f32.f32 %0, %1, 0f00000000;" : "=f"(m) : "f"(d)); return m;
}
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(dst)), "r"(ncols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(taddr), "r"(ncols) : "memory");
}
// N consecutive 32-bit columns of this thread's TMEM lane
template <int N> __device__ __forceinline__ void tmem_st(uint32_t t, const float* v);
template <> __device__ __forceinline__ void tmem_st<16>(uint32_t t, const float* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};"
                 :: "r"(t), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "f"(v[8]), "f"(v[9]),
                    "f"(v[10]), "f"(v[11]), "f"(v[12]), "f"(v[13]), "f"(v[14]), "f"(v[15]) : "memory");
}
template <> __device__ __forceinline__ void tmem_st<8>(uint32_t t, const float* v) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"
                 :: "r"(t), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}
// (the registers hold the columns after tmem_wait_ld, through which they pass, so that no use is moved ahead of it)
__device__ __forceinline__ void tmem_ld(uint32_t t, float (&v)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]),
                   "=f"(v[8]), "=f"(v[9]), "=f"(v[10]), "=f"(v[11]), "=f"(v[12]), "=f"(v[13]), "=f"(v[14]), "=f"(v[15]) : "r"(t) : "memory");
}
__device__ __forceinline__ void tmem_ld(uint32_t t, float (&v)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(t) : "memory");
}
template <int N> __device__ __forceinline__ void tmem_wait_ld(float (&v)[N]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < N; i += 8)
        asm volatile("" : "+f"(v[i]), "+f"(v[i + 1]), "+f"(v[i + 2]), "+f"(v[i + 3]), "+f"(v[i + 4]), "+f"(v[i + 5]), "+f"(v[i + 6]), "+f"(v[i + 7]));
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ int ld_relaxed(const int* p) {
    int v; asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory"); return v;
}
__device__ __forceinline__ unsigned long long ld_relaxed64(const void* p) {
    unsigned long long v; asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory"); return v;
}
__device__ __forceinline__ float4 ld_relaxed_f4(const float* p) {
    float4 v;
    asm volatile("ld.relaxed.gpu.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_relaxed_f(float* p, float v) {
    asm volatile("st.relaxed.gpu.global.f32 [%0], %1;" :: "l"(p), "f"(v) : "memory");
}
__device__ __forceinline__ float nonzero_f(float x) { return x == 0.f ? -0.f : x; }
__device__ __forceinline__ bool there(float4 v) {
    return __float_as_uint(v.x) != 0u && __float_as_uint(v.y) != 0u && __float_as_uint(v.z) != 0u && __float_as_uint(v.w) != 0u;
}
__device__ __forceinline__ bool there(double x) { return __double_as_longlong(x) != 0ll; }
__device__ __forceinline__ void red_or(int32_t* p, int v) {
    asm volatile("red.relaxed.gpu.global.or.b32 [%0], %1;" :: "l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void give_up(const StreamArgs& a, Shared& S) {
    atomicExch(a.wait_failed, 1);
    *(volatile int*)&S.failed = 1;
    *(volatile int*)&S.abort = 1;
}
__device__ __forceinline__ bool aborted(const Shared& S) { return *(volatile const int*)&S.abort != 0; }
// one more round of a wait for another CTA?  (sleeps; false: the bound has run out, or somebody has given up)
__device__ __forceinline__ bool wait_more(const StreamArgs& a, Shared& S, uint32_t i, unsigned ns) {
    if (i >= kSpin || aborted(S) || ((i & 63u) == 63u && ld_relaxed(a.wait_failed))) { give_up(a, S); return false; }
    __nanosleep(ns);
    return true;
}

// ------------------------------------------------------------------ merged rows
// Merge the T slice records of the rows of `unit` (a full warp; lane l takes slices l, l + 32, ...).  The records'
// sums are scaled to the largest exponent by powers of two (exactly) and added in one fixed order, so every
// warp that merges the same records gets the same bits.  Waits (bounded) for records not there yet: the next look is on its
// way before the last one has come back (a look takes 2,000 cycles under load; one at a time, two or three of them were
// most of the exchange).
template <int SPL>
__device__ __forceinline__ void merge_rows_n(const StreamArgs& a, Shared& S, int unit, Row* out_p, Row* out_q) {
    const int lane = threadIdx.x & 31, T = a.T;
    const Rec* base = a.rec + ((int64_t)unit * T) * 2;
    Rec r[SPL][2];
    if (SPL == 1) {
        const bool in = lane < T;
        const Rec* const p = base + 2 * (in ? lane : 0);
        Rec x[2], y[2];
        x[0] = ld_cg(p); x[1] = ld_cg(p + 1);
        for (uint32_t i = 0;; ++i) {
            __nanosleep(S_LOOK);
            y[0] = ld_cg(p); y[1] = ld_cg(p + 1);
            if (__all_sync(0xffffffffu, rec_valid(x[0]) && rec_valid(x[1]))) break;
            x[0] = y[0]; x[1] = y[1];
            if (i >= kSpin || aborted(S) || ((i & 63u) == 63u && ld_relaxed(a.wait_failed))) { give_up(a, S); break; }
        }
#pragma unroll
        for (int w = 0; w < 2; ++w) r[0][w] = in && rec_valid(x[w]) ? x[w] : no_rec();
    } else {
        unsigned missing = 0;
#pragma unroll
        for (int i = 0; i < SPL; ++i)
#pragma unroll
            for (int w = 0; w < 2; ++w) { r[i][w] = no_rec(); if (lane + 32 * i < T) missing |= 1u << (2 * i + w); }
        for (uint32_t it = 0;; ++it) {
#pragma unroll
            for (int i = 0; i < SPL; ++i)
#pragma unroll
                for (int w = 0; w < 2; ++w)
                    if (missing & (1u << (2 * i + w))) {
                        const Rec x = ld_cg(base + 2 * (lane + 32 * i) + w);
                        if (rec_valid(x)) { r[i][w] = x; missing &= ~(1u << (2 * i + w)); }
                    }
            if (!__any_sync(0xffffffffu, missing != 0) || !wait_more(a, S, it, 100)) break;
        }
    }
#pragma unroll
    for (int w = 0; w < 2; ++w) {
        int el = E_EMPTY, bad = 0;
#pragma unroll
        for (int i = 0; i < SPL; ++i) { el = max(el, rec_e(r[i][w])); bad |= r[i][w].flags & 1; }
        const int Em = redux_max(el);
        double v = 0.0;
#pragma unroll
        for (int i = 0; i < SPL; ++i) { const int e = rec_e(r[i][w]); if (e > E_EMPTY) v += r[i][w].s * pow2d(max(e - Em, -1000)); }
        v = warp_sum(v);
        Row x;
        x.st = __any_sync(0xffffffffu, bad) || !(v == v) ? ST_NONFINITE : Em == E_EMPTY ? ST_EMPTY : 0;
        x.inv_s = !x.st && v > 0.0 ? 1.0 / v : 0.0; x.e = Em;
        if (w == 0) *out_p = x; else *out_q = x;
    }
}
struct Rows { Row p, q; };
__device__ __noinline__ Rows merge_rows_long(const StreamArgs& a, Shared& S, int unit) {
    Rows r;
    merge_rows_n<kStreamMaxSlices / 32>(a, S, unit, &r.p, &r.q);
    return r;
}

// rho = S_p / S_q as two floats; pass 2 forms r' = max(0, e_p - rho e_q) = (p - q) S_p 2^(E_p - E_wp)
struct Scale { float rho_h, rho_l; int ep, eq; };
__device__ __forceinline__ Scale scale_of(const Row& rp, const Row& rq) {
    Scale sc;
    const double rho = rp.inv_s > 0.0 ? rq.inv_s / rp.inv_s : 0.0;
    sc.rho_h = (float)rho; sc.rho_l = (float)(rho - (double)sc.rho_h);
    sc.ep = rp.st ? E_EMPTY : rp.e; sc.eq = rq.st ? E_EMPTY : rq.e;
    return sc;
}
// the chunk's rho: e_p sits around E_wp, e_q around E_wq, so rho takes the factor 2^((E_wq - E_rq) - (E_wp - E_rp))
// (exact; a chunk whose target or draft part is empty has no such factor: its e are all zero); z, w: the factors that
// bring the chunk's r' and e_q to the rows' exponents
__device__ __forceinline__ float4 chunk_rho(const Scale& sc, int ewp, int ewq) {
    int k = 0;
    if (ewp > E_EMPTY && ewq > E_EMPTY && sc.ep > E_EMPTY && sc.eq > E_EMPTY) k = (ewq - sc.eq) - (ewp - sc.ep);
    k = max(min(k, 126), -126);
    const float f = pow2f(k);
    return make_float4(sc.rho_h * f, sc.rho_l * f,
                       ewp > E_EMPTY && sc.ep > E_EMPTY ? pow2f(max(ewp - sc.ep, -127)) : 0.f,
                       ewq > E_EMPTY && sc.eq > E_EMPTY ? pow2f(max(ewq - sc.eq, -127)) : 0.f);
}

// ------------------------------------------------------------------ producer
// One thread.  A sequence has `tps` tasks: slice s of row pair k for k = 0 .. K - 1, s = 0 .. T - 1, then the bonus
// row two slices at a time; CTA i takes the tasks i, i + grid, ... and skips those of positions past the sequence's
// draft length.  What the next task needs from memory (draft length, temperature) is asked for one task ahead.
// A task's two rows take a stage each.
struct Next { int t, b, k, s, L, bonus; float tau; };
template <bool TVM>
__device__ __forceinline__ Next fetch_next(const StreamArgs& a, int t) {
    const RowArgs& R = a.r;
    Next x;
    x.t = t;
    x.b = t / a.tps;
    const int r = t - x.b * a.tps;
    x.L = TVM ? 1 : len_of(R, x.b);
    x.tau = tau_of(R, x.b);
    const int npair = TVM ? a.tps : R.K * a.T;
    if (r < npair) { x.k = r / a.T; x.s = r - x.k * a.T; x.bonus = 0; }
    else { x.k = x.L; x.s = 2 * (r - npair); x.bonus = 1; }
    return x;
}
struct Producer { Next nx; long long t; int n, u, st; const char* src; uint32_t bytes; };    // u: stages filled so far, st = u % NSTG
// fill the next stage; FIRST: one of the first NSTG, free from the start.  False: no task is left.
template <int DT, bool TVM, bool FIRST>
__device__ __noinline__ bool produce(const StreamArgs& a, Shared& S, uint32_t data, Producer& P) {
    const RowArgs& R = a.r;
    const uint32_t par = ((uint32_t)(P.u / NSTG) & 1u) ^ 1u;
    if (!(P.u & 1)) {
        Next cur;
        do {
            cur = P.nx;
            if (cur.t < 0) return false;
            P.t += gridDim.x;
            if (P.t < a.total) P.nx = fetch_next<TVM>(a, (int)P.t); else P.nx.t = -1;
        } while (!TVM && !cur.bonus && cur.k >= cur.L);              // positions past the sequence's draft length
        const int v0 = cur.s * a.slice_vecs, nv = min(a.slice_vecs, R.nvec - v0);
        const int v1 = cur.bonus ? v0 + a.slice_vecs : v0, nv1 = cur.bonus ? (cur.s + 1 < a.T ? min(a.slice_vecs, R.nvec - v1) : 0) : nv;
        const bool tail = R.V % Elem<DT>::VEC != 0 && (v0 + nv == R.nvec || (nv1 > 0 && v1 + nv1 == R.nvec));
        const char* row = row_ptr(R, cur.b, cur.k);
        Task d;
        d.unit = cur.b * a.ups + cur.k;
        d.us = d.unit * a.T + cur.s;
        d.c = temp_scale(cur.tau).hi;
        d.meta = (cur.bonus ? kBonus : kPair) | (nv << 2) | (nv1 << 14) | (tail ? 1 << 26 : 0);
        if (!FIRST && !mbar_wait<S_EMPTY>(S, smem_u32(&S.empty[P.st]), par)) { give_up(a, S); return false; }
        S.task[P.n % RT] = d;
        ++P.n;
        mbar_arrive_expect(&S.full[P.st], (uint32_t)nv * 16u);
        bulk_load(data + P.st * STAGE, row + (int64_t)v0 * 16, (uint32_t)nv * 16u, &S.full[P.st]);
        P.src = (cur.bonus ? row : row_ptr(R, cur.b, R.K + 1 + cur.k)) + (int64_t)v1 * 16;
        P.bytes = (uint32_t)nv1 * 16u;
    } else {
        if (!FIRST && !mbar_wait<S_EMPTY>(S, smem_u32(&S.empty[P.st]), par)) { give_up(a, S); return false; }
        if (P.bytes) { mbar_arrive_expect(&S.full[P.st], P.bytes); bulk_load(data + P.st * STAGE, P.src, P.bytes, &S.full[P.st]); }
        else mbar_arrive(&S.full[P.st]);
    }
    ++P.u;
    if (++P.st == NSTG) P.st = 0;
    return true;
}
// The end of the tasks, marked in as many descriptions as there are stats warps.  Nothing is in flight when this returns, also
// when somebody has given up.
__device__ __forceinline__ void produce_stop(const StreamArgs& a, Shared& S, const Producer& P) {
    int u = max(P.u - NSTG, 0);
    if (!aborted(S) && mbar_wait<S_EMPTY>(S, smem_u32(&S.empty[P.st]), ((uint32_t)(P.u / NSTG) & 1u) ^ 1u)) {
        for (int i = 0; i < NSTAT; ++i) S.task[(P.n + i) % RT].meta = kStop;
        mbar_arrive(&S.full[P.st]);
        u = max(P.u - NSTG + 1, 0);          // (the stage that the mark took had been read: its barrier is a turn further)
    }
    for (; u < P.u; ++u)
        for (uint32_t i = 0; i < kWaitSpin && !mbar_try(smem_u32(&S.full[u % NSTG]), (uint32_t)(u / NSTG) & 1u); ++i) {}
}

// ------------------------------------------------------------------ consumers
__device__ __forceinline__ float2 add_pairs(float2 acc, const float* e, int n) {
#pragma unroll
    for (int i = 0; i < n; i += 2) acc = __fadd2_rn(acc, make_float2(e[i], e[i + 1]));
    return acc;
}
// Residuals of N token pairs from their exponentials: d = e_p - rho e_q, rho as two floats (equal rows give rho = 1
// and d = 0 exactly), r' = max(0, d).  As e_p <= 1, d saturated to [0, 1] is max(0, d): one fused multiply-add.
// Adds the sum of the r' to *tm; with R, leaves the r'.
template <int N, bool R>
__device__ __forceinline__ void resid_n(const float* ep, const float* eq, float h, float l, float2* tm, float* r) {
    const float2 nl = make_float2(-l, -l);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 t = __ffma2_rn(nl, make_float2(eq[i], eq[i + 1]), make_float2(ep[i], ep[i + 1]));
        const float2 d = make_float2(fma_sat(-h, eq[i], t.x), fma_sat(-h, eq[i + 1], t.y));
        if (R) { r[i] = d.x; r[i + 1] = d.y; }
        *tm = __fadd2_rn(*tm, d);
    }
}
// ... with the sum of e_q over the pairs with d >= 0 (q <= p) in *sx: the mask 1[d >= 0] serves both sums
template <int N>
__device__ __forceinline__ void resid_aux_n(const float* ep, const float* eq, float h, float l, float2* tm, float2* sx) {
    const float2 nh = make_float2(-h, -h), nl = make_float2(-l, -l);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 q2 = make_float2(eq[i], eq[i + 1]);
        const float2 d = __ffma2_rn(nh, q2, __ffma2_rn(nl, q2, make_float2(ep[i], ep[i + 1])));
        const float2 mk = make_float2(set_ge0(d.x), set_ge0(d.y));
        *tm = __ffma2_rn(d, mk, *tm);
        *sx = __ffma2_rn(q2, mk, *sx);
    }
}
// lanes 0..15 get the warp's sum of p, lanes 16..31 that of q
__device__ __forceinline__ float warp_sum2(float p, float q, bool hi) {
    float x = hi ? q : p;
    const float y = hi ? p : q;
    x += __shfl_xor_sync(0xffffffffu, y, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}
template <int DT> __device__ __forceinline__ float vecs_max(const uint4* v) {
    return max_nan(max_nan(vec_max<DT>(v[0]), vec_max<DT>(v[1])), max_nan(vec_max<DT>(v[2]), vec_max<DT>(v[3])));
}
template <> __device__ __forceinline__ float vecs_max<1>(const uint4* v) {
    uint32_t a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) a[j] = max_nan_bf16x2(max_nan_bf16x2(v[j].x, v[j].y), max_nan_bf16x2(v[j].z, v[j].w));
    const uint32_t m = max_nan_bf16x2(max_nan_bf16x2(a[0], a[1]), max_nan_bf16x2(a[2], a[3]));
    return max_nan(__uint_as_float(m << 16), __uint_as_float(m & 0xffff0000u));
}

// Where a chunk's exponentials wait for pass 2: vector j's, target row then draft row, in TMEM columns; MIX: the last
// two vectors' in shared memory.
template <int DT, bool MIX> __device__ __forceinline__ void park(uint32_t tcol, uint32_t msl, int j, const float* v) {
    constexpr int N = 2 * Elem<DT>::VEC;
    if (MIX && j >= 2) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) sts16(msl + ((j - 2) * (N / 4) + i) * 512, v + 4 * i);
    } else tmem_st<N>(tcol + j * N, v);
}
// (from TMEM: in the registers after tmem_wait_ld)
template <int DT, bool MIX, int N> __device__ __forceinline__ void fetch(uint32_t tcol, uint32_t msl, int j, float (&v)[N]) {
    if (MIX && j >= 2) {
#pragma unroll
        for (int i = 0; i < N / 4; ++i) {
            const float4 u = lds16f(msl + ((j - 2) * (N / 4) + i) * 512);
            v[4 * i] = u.x; v[4 * i + 1] = u.y; v[4 * i + 2] = u.z; v[4 * i + 3] = u.w;
        }
    } else tmem_ld(tcol + j * N, v);
}
template <int N, bool TVM> __device__ __forceinline__ void resid(const float* p, const float* r, float4 rho, float2& tm, float2& sx) {
    if (TVM) resid_aux_n<N>(p, r, rho.x, rho.y, &tm, &sx);
    else resid_n<N, false>(p, r, rho.x, rho.y, &tm, nullptr);
}
// A full chunk of both rows (p0, p1: the lane's first vectors in the stages) and pass 2 of the task before in its place.
// The logits are read twice from shared memory, for the largest and for the exponentials: kept in registers they
// were spilled, and with all but 20 KB of the SM's memory taken as shared, spills go to L2.
template <int DT, bool TVM, bool MIX>
__device__ __forceinline__ void both_passes(uint32_t tcol, uint32_t msl, uint32_t p0, uint32_t p1, float c, float efp, float efq,
                                            float4 rho, float2& ap, float2& aq, float2& tm, float2& sx) {
    constexpr int VEC = Elem<DT>::VEC;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float v[2 * VEC], e[2 * VEC];
        const uint4 x = lds16(p0 + j * 512), y = lds16(p1 + j * 512);
        fetch<DT, MIX>(tcol, msl, j, v);
        exp_vec<DT>(x, c, efp, e);
        exp_vec<DT>(y, c, efq, e + VEC);
        if (!(MIX && j >= 2)) tmem_wait_ld(v);
        resid<VEC, TVM>(v, v + VEC, rho, tm, sx);
        ap = add_pairs(ap, e, VEC);
        aq = add_pairs(aq, e + VEC, VEC);
        park<DT, MIX>(tcol, msl, j, e);
    }
}
template <int DT, bool TVM>
__device__ __forceinline__ void pass2(bool mix, uint32_t tcol, uint32_t msl, float4 rho, float2& tm, float2& sx) {
    constexpr int VEC = Elem<DT>::VEC;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float v[2 * VEC];
        if (mix && j >= 2) fetch<DT, true>(tcol, msl, j, v); else { fetch<DT, false>(tcol, msl, j, v); tmem_wait_ld(v); }
        resid<VEC, TVM>(v, v + VEC, rho, tm, sx);
    }
}
template <int DT>
__device__ __forceinline__ void pass1(bool mix, bool keep, uint32_t tcol, uint32_t msl, const uint4* xp, const uint4* xq, float c, float efp, float efq,
                                      float2& ap, float2& aq) {
    constexpr int VEC = Elem<DT>::VEC;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float e[2 * VEC];
        exp_vec<DT>(xp[j], c, efp, e);
        exp_vec<DT>(xq[j], c, efq, e + VEC);
        ap = add_pairs(ap, e, VEC);
        aq = add_pairs(aq, e + VEC, VEC);
        if (keep) { if (mix && j >= 2) park<DT, true>(tcol, msl, j, e); else park<DT, false>(tcol, msl, j, e); }
    }
}

// A consumer warp.  Step n: pass 1 of its chunk of both rows of task n and pass 2 of task n - NSLOT, whose place task n
// takes: a vector's exponentials are read before those of the new task are put there.  Both rows and both passes in one
// step: the chains of dependent instructions around the arithmetic (barrier, description, largest logit, sums) are
// as long as the arithmetic itself and are met once per task.  The warps do not wait for each other.
template <int DT, bool TVM>
__device__ __forceinline__ void consumer(const StreamArgs& a, SharedD<DT>& S, uint32_t data, int tid) {
    using D = Dims<DT>;
    constexpr int VEC = D::VEC, NSLOT = D::NSLOT;
    const int lane = tid & 31, w = tid >> 5;
    const bool one = lane == 0;
    // the warp's columns of its quarter of the lanes
    const uint32_t tbase = S.tmem_base + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((w >> 2) * D::WCOL);
    const uint32_t mine = data + (w * CV + lane) * 16;
    const uint32_t msl = data + RING + w * D::MWARP + lane * 16;
    const uint32_t full0 = smem_u32(S.full), empty0 = smem_u32(S.empty), task0 = smem_u32(S.task);
    uint32_t st = 0, par = 0;                         // stage of the next row, parity of its turn
    int n_end = 0x7fffff00;                           // the first step without a task
    int slot = 0;                                     // n % NSLOT
#pragma unroll 1
    for (int n = 0; n < n_end + NSLOT; ++n) {
        bool live = n < n_end;
        const bool live2 = n >= NSLOT;
        const int m = n - NSLOT;
        float c = 0.f;
        int meta = kStop;
        uint32_t p0 = 0, p1 = 0, e0 = 0, e1 = 0;
        if (live) {
            if (!mbar_wait<S_FULL>(S, full0 + st * 8, par)) { if (one) give_up(a, S); return; }
            const uint4 d = lds16(task0 + (n % RT) * 16);
            c = __uint_as_float(d.x); meta = (int)d.y;
            if (t_kind(meta) == kStop) {
                n_end = n; live = false;
                if (one) for (int i = 0; i < NSTAT; ++i) mbar_arrive(&S.pdone[(n + i) % R8]);       // every stats warp meets the end
            } else {
                p0 = mine + st * STAGE; e0 = empty0 + st * 8;
                if (++st == NSTG) { st = 0; par ^= 1u; }
                if (!mbar_wait<S_FULL>(S, full0 + st * 8, par)) { if (one) give_up(a, S); return; }
                p1 = mine + st * STAGE; e1 = empty0 + st * 8;
                if (++st == NSTG) { st = 0; par ^= 1u; }
            }
        }
        int meta2 = kStop, us2 = 0;
        float4 rho = make_float4(0.f, 0.f, 0.f, 0.f);
        bool two = false;                              // there is pass 2 to do
        if (live2) {
            if (!mbar_wait<S_STAT>(S, smem_u32(&S.stats[m % R8]), (m / R8) & 1u)) { if (one) give_up(a, S); return; }
            const uint4 d = lds16(task0 + (m % RT) * 16);
            meta2 = (int)d.y; us2 = (int)d.z;
            two = t_kind(meta2) == kPair && w * CV < t_nv(meta2);
            if (two) rho = S.slot[slot].rho[w];
            tmem_wait_st();
        }
        const int left0 = live ? t_nv(meta) - w * CV : 0, left1 = live ? t_nv2(meta) - w * CV : 0;     // vectors from the chunk's first to the end of the slice
        const bool mix = D::MWARP != 0 && slot == NSLOT - 1;
        const uint32_t tcol = tbase + slot * D::TCOL;
        QExp Ep, Eq;
        Ep.e = E_EMPTY; Ep.ef = 0.f; Eq.e = E_EMPTY; Eq.ef = 0.f;
        float2 ap = make_float2(0.f, 0.f), aq = ap, tm = ap, sx = ap;
        if (two && left1 >= CV && t_kind(meta) == kPair && !t_tail(meta)) {
            // the usual step, without a branch inside, so that the compiler deals the exponentials out among the rest
            uint4 x[4], y[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = lds16(p0 + j * 512);
#pragma unroll
            for (int j = 0; j < 4; ++j) y[j] = lds16(p1 + j * 512);
            Ep = chunk_exponent(vecs_max<DT>(x), c);
            Eq = chunk_exponent(vecs_max<DT>(y), c);
            if (!mix) both_passes<DT, TVM, false>(tcol, msl, p0, p1, c, Ep.ef, Eq.ef, rho, ap, aq, tm, sx);
            else both_passes<DT, TVM, true>(tcol, msl, p0, p1, c, Ep.ef, Eq.ef, rho, ap, aq, tm, sx);
        } else {
            if (two) pass2<DT, TVM>(mix, tcol, msl, rho, tm, sx);
            if (left0 > 0) {                           // (the second row is never the longer one)
                uint4 xp[4], xq[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) { xp[j] = lds16(p0 + j * 512); xq[j] = lds16(p1 + j * 512); }
                if (left1 < CV || t_tail(meta)) {
                    // not a full chunk: vectors beyond the slice read as -inf, a row's ragged last vector loses the lanes beyond the vocabulary
                    const int lastn = a.r.V - (a.r.nvec - 1) * VEC;
                    const bool tp = t_tail(meta) && (t_kind(meta) == kPair || t_nv2(meta) == 0), tq = t_tail(meta);
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int vi = j * 32 + lane;
                        if (vi >= left0) xp[j] = neg_inf_vec<DT>();
                        if (vi >= left1) xq[j] = neg_inf_vec<DT>();
                        if (tp && vi == left0 - 1) mask_tail<DT>(xp[j], lastn);
                        if (tq && vi == left1 - 1) mask_tail<DT>(xq[j], lastn);
                    }
                }
                Ep = chunk_exponent(vecs_max<DT>(xp), c);
                Eq = chunk_exponent(vecs_max<DT>(xq), c);
                pass1<DT>(mix, t_kind(meta) == kPair, tcol, msl, xp, xq, c, Ep.ef, Eq.ef, ap, aq);       // (a bonus task's exponentials are summed and not kept)
            }
        }
        if (live) {
            __syncwarp();
            if (one) { mbar_arrive(e0); mbar_arrive(e1); }
        }
        if (live) {
            const int2 s0 = warp_sum_words(ap.x + ap.y), s1 = warp_sum_words(aq.x + aq.y);
            if (one) {
                S.slot[slot].part[0][w] = make_int4(s0.x, s0.y, Ep.e, 0);
                S.slot[slot].part[1][w] = make_int4(s1.x, s1.y, Eq.e, 0);
                mbar_arrive(&S.pdone[n % R8]);
            }
        }
        if (t_kind(meta2) == kPair) {
            const int64_t o = (int64_t)us2 * CH + w;
            if (TVM) {
                const float z = warp_sum2(tm.x + tm.y, sx.x + sx.y, lane >= 16) * (lane >= 16 ? rho.w : rho.z);
                if ((lane & 15) == 0) st_relaxed_f((lane ? a.ca : a.cm) + o, nonzero_f(z));
            } else {
                const float z = warp_sum(tm.x + tm.y) * rho.z;
                if (one) st_relaxed_f(a.cm + o, nonzero_f(z));
            }
        }
        if (++slot == NSLOT) slot = 0;
        __syncwarp();
    }
}

// ------------------------------------------------------------------ stats warps
// Stats warp j serves the tasks n = j, j + NSTAT, ...  Lane l takes chunk l % 16 of the target row (l < 16) or of the
// draft row: the chunks' sums, in fixed point around the chunks' exponents, are shifted to the slice's largest exponent
// and added, and the slice's records are stored.  A bonus task ends there: its chunk sums, around their slice's exponent,
// are the masses of the draw.  For a row pair the warp then finds the T records of the unit, merges both rows and leaves
// each chunk's rho; with slice 0 go the merged rows, for the warp that completes the sequence.
struct Part { double s; unsigned ub; int em; bool bad; };
__device__ __forceinline__ Part slice_part(long long n, int ew) {
    Part r;
    r.em = redux_max(ew);
    r.bad = r.em >= E_BAD;
    if (r.bad) r.em = E_EMPTY;
    const bool in = ew > E_EMPTY && !r.bad;
    const int d = in ? min(r.em - ew, 62) : 0;
    const long long v = in ? n >> d : 0;                    // below 2^50; what is shifted out is below 2^-40 each
    const unsigned hi = (unsigned)(v >> 26), lo = (unsigned)v & 0x3ffffffu;
    const unsigned long long t = ((unsigned long long)(unsigned)redux_add((int)hi) << 26) + (unsigned)redux_add((int)lo);
    r.s = (double)t * 9.094947017729282e-13;                // 2^-40
    // 4^(E_w - E_s) times the chunk's sum of e, in units of 2^-14, rounded up
    r.ub = (unsigned)redux_add(in ? (int)((hi >> min(d, 31)) + 1u) : 0);
    return r;
}
template <int DT>
__device__ __noinline__ void stats_warp(const StreamArgs& a, SharedD<DT>& S, int j) {
    const int lane = threadIdx.x & 31, row = lane >> 4, chunk = lane & 15;
#pragma unroll 1
    for (int n = j;; n += NSTAT) {
        if (!mbar_wait<S_PD>(S, smem_u32(&S.pdone[n % R8]), ((uint32_t)(n / R8)) & 1u)) { if (lane == 0) give_up(a, S); return; }
        const int meta = S.task[n % RT].meta, us = S.task[n % RT].us, unit = S.task[n % RT].unit;
        if (t_kind(meta) == kStop) return;
        const bool pair = t_kind(meta) == kPair;
        Slot& sl = S.slot[n % Dims<DT>::NSLOT];
        int4 c = sl.part[row][min(chunk, CH - 1)];
        if (chunk >= CH) c = make_int4(kNoSum0, kNoSum1, E_EMPTY, 0);     // (lanes without a chunk)
        const long long ns = words_sum(c.x, c.y);
        const Part p0 = slice_part(ns, row ? E_EMPTY : c.z), p1 = slice_part(ns, row ? c.z : E_EMPTY);
        const bool two = t_nv2(meta) > 0;                   // a second record: the draft row's, or the bonus row's second slice's
        {
            // Every lane forms the record; lanes 0 and 16 store it, by predicate (as a branch for those two lanes the
            // store comes late: nothing makes a warp that has split reconverge before its next __syncwarp()).
            const unsigned long long w0 = (unsigned long long)__double_as_longlong(nonzero_bits(row ? p1.s : p0.s));
            const float ub = (float)(row ? p1.ub : p0.ub) * 6.103515625e-05f;                // 2^-14; below 2^24 units: exact
            const unsigned ubits = ((unsigned)__float_as_int(ub) + 1u) & ~1u;                // (bit 0 is the flag)
            const unsigned long long w1 = (unsigned long long)(unsigned)rec_code(row ? p1.em : p0.em)
                                        | ((unsigned long long)(ubits | ((row ? p1.bad : p0.bad) ? 1u : 0u)) << 32);
            const unsigned doit = (chunk == 0 && (row == 0 || two)) ? 1u : 0u;
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};\n\t}"
                         :: "l"(a.rec + (int64_t)us * 2 + (row ? (pair ? 1 : 2) : 0)), "l"(w0), "l"(w1), "r"(doit) : "memory");
        }
        if (!pair) {
            const Part& p = row ? p1 : p0;
            const float m = c.z > E_EMPTY && !p.bad ? (float)ns * 9.094947017729282e-13f * pow2f(max(c.z - p.em, -127)) : 0.f;
            if (chunk < CH && (row == 0 || two)) st_relaxed_f(a.cm + (int64_t)(us + row) * CH + chunk, nonzero_f(m));
            __syncwarp();
            if (lane == 0) mbar_arrive(&S.stats[n % R8]);
            __syncwarp();
            continue;
        }
        if (a.expire == 2) { if (lane == 0) give_up(a, S); return; }       // test hook: this wait's bound has run out already
        Row rp, rq;
        if (a.T <= 32) merge_rows_n<1>(a, S, unit, &rp, &rq);
        else { const Rows r = merge_rows_long(a, S, unit); rp = r.p; rq = r.q; }
        const Scale sc = scale_of(rp, rq);
        const int exq = __shfl_xor_sync(0xffffffffu, c.z, 16);
        if (row == 0 && chunk < CH) sl.rho[chunk] = chunk_rho(sc, c.z, exq);
        __syncwarp();
        if (lane == 0) mbar_arrive(&S.stats[n % R8]);
        if (lane < 2 && us == unit * a.T) {
            Row x = lane ? rq : rp;
            x.inv_s = nonzero_bits(x.inv_s); x.st |= kRowValid;
            st16(a.rows + 2 * (int64_t)unit + lane, x);
        }
        __syncwarp();
    }
}

// ------------------------------------------------------------------ completing sequences
__device__ __forceinline__ Row wait_row(const StreamArgs& a, Shared& S, const Row* p) {
    Row x = ld_cg(p);
    for (uint32_t i = 0; !rec_valid(x); ++i) {
        if (!wait_more(a, S, i, 100)) { x.inv_s = 0.0; x.e = E_EMPTY; x.st = ST_WAIT; break; }
        x = ld_cg(p);
    }
    x.st &= 0xff;
    return x;
}
__device__ __forceinline__ Rec wait_rec(const StreamArgs& a, Shared& S, const Rec* p) {
    Rec x = ld_cg(p);
    for (uint32_t i = 0; !rec_valid(x); ++i) {
        if (!wait_more(a, S, i, 100)) return no_rec();
        x = ld_cg(p);
    }
    return x;
}
__device__ __forceinline__ Row shfl_row(const Row& x, int src) {
    Row y;
    y.inv_s = __shfl_sync(0xffffffffu, x.inv_s, src); y.e = __shfl_sync(0xffffffffu, x.e, src); y.st = __shfl_sync(0xffffffffu, x.st, src);
    return y;
}
__device__ __forceinline__ double sum4(float4 v) { return ((double)v.x + (double)v.y) + ((double)v.z + (double)v.w); }
// The sum of the lane's run [i0, i1) of a unit's chunk masses (four at a time); waits (bounded) for those not there yet.
// Four loads are on their way at once.
__device__ __forceinline__ double run_masses(const StreamArgs& a, Shared& S, const float* m, int i0, int i1) {
    double z = 0.0;
    for (int i = i0; i < i1; i += 4) {
        float4 v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { v[k] = make_float4(-0.f, -0.f, -0.f, -0.f); if (i + k < i1) v[k] = ld_relaxed_f4(m + 4 * (i + k)); }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            for (uint32_t t = 0; !there(v[k]) && wait_more(a, S, t, 100); ++t) v[k] = ld_relaxed_f4(m + 4 * (i + k));
            z += sum4(v[k]);
        }
    }
    return z;
}
// the wait for a sequence's turn: long sleeps until its last row pair's normalisers are there
__device__ __forceinline__ void wait_turn(const StreamArgs& a, Shared& S, const Row* p) {
    for (uint32_t i = 0; !rec_valid(ld_cg(p)); ++i) if (!wait_more(a, S, i, 400)) return;
}

// bebop_tv: row pair b is complete when its chunks' masses are in
__device__ __noinline__ void finish_tv(const StreamArgs& a, Shared& S, int b) {
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, n4 = a.T * (CH / 4), per = (n4 + 31) / 32;
    const int i0 = min(lane * per, n4), i1 = min(i0 + per, n4);
    wait_turn(a, S, a.rows + 2 * (int64_t)b);
    const Row rp = wait_row(a, S, a.rows + 2 * (int64_t)b), rq = wait_row(a, S, a.rows + 2 * (int64_t)b + 1);
    const int st = tau_ok(tau_of(R, b)) ? (rp.st | rq.st) : ST_BAD_TEMP;
    double z = 0.0, sx = 0.0;
    if (!st) {
        z = warp_sum(run_masses(a, S, a.cm + (int64_t)b * a.T * CH, i0, i1)) * rp.inv_s;
        if (a.s_aux) sx = warp_sum(run_masses(a, S, a.ca + (int64_t)b * a.T * CH, i0, i1)) * rq.inv_s;
    }
    if (lane == 0) {
        a.o.tv[b] = (float)fmin(fmax(z, 0.0), 1.0);
        if (a.s_aux) a.s_aux[b] = (float)sx;
        if (a.o.row_status && st) red_or(a.o.row_status + b, st);
    }
}

// four chunk masses of a bonus row: each slice's chunks stand around the slice's exponent
__device__ __forceinline__ float4 bonus4(const StreamArgs& a, Shared& S, int unit, int i4, int erow) {
    const float* m = a.cm + (int64_t)unit * a.T * CH + 4 * i4;
    float4 v = ld_relaxed_f4(m);
    const int e = rec_e(wait_rec(a, S, a.rec + ((int64_t)unit * a.T + i4 / (CH / 4)) * 2));
    for (uint32_t t = 0; !there(v) && wait_more(a, S, t, 100); ++t) v = ld_relaxed_f4(m);
    const float f = e > E_EMPTY ? pow2f(max(e - erow, -127)) : 0.f;
    v.x *= f; v.y *= f; v.z *= f; v.w *= f;
    return v;
}
// the r' (or, without a draft row, the e) of one vector, as pass 1 and pass 2 of the sweep formed them
template <int DT>
__device__ __forceinline__ void draw_vec(const uint4& vp, const uint4& vq, bool pair, float c, const QExp& Ep, const QExp& Eq, float4 rho, float* r) {
    constexpr int VEC = Elem<DT>::VEC;
    float ep[VEC], eq[VEC];
    exp_vec<DT>(vp, c, Ep.ef, ep);
    if (pair) {
        float2 t = make_float2(0.f, 0.f);
        exp_vec<DT>(vq, c, Eq.ef, eq);
        resid_n<VEC, true>(ep, eq, rho.x, rho.y, &t, r);
    } else {
#pragma unroll
        for (int i = 0; i < VEC; ++i) r[i] = ep[i];
    }
}

// bebop_verify: one warp completes sequence b.  The accept scan runs as soon as the rows' normalisers are there, two tasks
// ahead of the masses, so that what follows the last mass is short: the draw unit's masses -> the owning lane's
// chunks -> the owning chunk's vectors.
template <int DT>
__device__ __noinline__ void finish_seq(const StreamArgs& a, Shared& S, int b) {
    constexpr int VEC = Elem<DT>::VEC;
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31;
    const int K = R.K, V = R.V, T = a.T, L = len_of(R, b);
    const float tau = tau_of(R, b);
    const TempScale ts = temp_scale(tau);
    int seq_st = tau_ok(tau) ? 0 : ST_BAD_TEMP;
    const int unit0 = b * (K + 1);
    // ---- lane k owns draft position k: its token, uniform and the token's logits are the call's inputs, asked for
    // before the wait for the sequence's turn
    const bool active = lane < L;
    const int tk = active ? a.draft_tokens[(int64_t)b * K + lane] : 0;
    const float u = active ? a.u_accept[(int64_t)b * K + lane] : 0.f;
    const float uf = a.u_final[b];
    const bool tok_ok = tk >= 0 && tk < V;
    float zpx = 0.f, zqx = 0.f;
    if (active && tok_ok) { zpx = load_one<DT>(row_ptr(R, b, lane), tk); zqx = load_one<DT>(row_ptr(R, b, K + 1 + lane), tk); }
    if (L > 0) wait_turn(a, S, a.rows + 2 * (int64_t)(unit0 + L - 1));
    // ---- its rows
    Row sp, sq;
    sp.inv_s = 0.0; sp.e = E_EMPTY; sp.st = 0; sq = sp;
    if (active) { sp = wait_row(a, S, a.rows + 2 * (int64_t)(unit0 + lane)); sq = wait_row(a, S, a.rows + 2 * (int64_t)(unit0 + lane) + 1); }
    if (!seq_st && __ballot_sync(0xffffffffu, active && !tok_ok)) seq_st = ST_BAD_TOKEN;
    const int rs = active ? (sp.st | sq.st) : 0;
    const unsigned badrows = __ballot_sync(0xffffffffu, rs != 0);
    const int first_bad = badrows ? __ffs(badrows) - 1 : 32;
    const int rs_first = __shfl_sync(0xffffffffu, rs, first_bad & 31);
    if (!seq_st && badrows) seq_st = rs_first;
    double px = 0.0, qx = 0.0;
    bool acc = false;
    if (active && !(seq_st & (ST_FATAL | ST_WAIT)) && lane < first_bad) {
        const double cd = (double)ts.hi;
        px = exp2((double)zpx * cd - (double)sp.e) * sp.inv_s;
        qx = exp2((double)zqx * cd - (double)sq.e) * sq.inv_s;
        acc = (double)u * qx < px;
    }
    const unsigned rej = __ballot_sync(0xffffffffu, active && !acc);
    const int n = rej ? __ffs(rej) - 1 : L;
    // ---- the bonus row, when every draft was accepted: merged here from its slices' records
    Row rb; rb.inv_s = 0.0; rb.e = E_EMPTY; rb.st = 0;
    if (!(seq_st & (ST_FATAL | ST_WAIT)) && n == L) {
        const Rec* base = a.rec + ((int64_t)(unit0 + L) * T) * 2;
        int el = E_EMPTY, bad = 0;
        for (int i = lane; i < T; i += 32) { const Rec r = wait_rec(a, S, base + 2 * i); bad |= r.flags & 1; el = max(el, rec_e(r)); }
        rb.e = redux_max(el);
        double v = 0.0;
        for (int i = lane; i < T; i += 32) { const Rec r = wait_rec(a, S, base + 2 * i); if (rec_e(r) > E_EMPTY) v += r.s * pow2d(max(rec_e(r) - rb.e, -1000)); }
        v = warp_sum(v);
        rb.st = __any_sync(0xffffffffu, bad) || !(v == v) ? ST_NONFINITE : rb.e == E_EMPTY ? ST_EMPTY : 0;
        rb.inv_s = !rb.st && v > 0.0 ? 1.0 / v : 0.0;
        seq_st |= rb.st;
    }
    if (__any_sync(0xffffffffu, aborted(S))) seq_st = ST_WAIT;
    const bool fatal = (seq_st & (ST_FATAL | ST_WAIT)) != 0;
    const int nn = fatal ? 0 : n;
    for (int q = lane; q <= K; q += 32)
        if (fatal || q != nn) a.o.out_tokens[(int64_t)b * (K + 1) + q] = q < nn ? tk : -1;
    if (lane < K) {
        const bool zero = fatal || lane >= L;
        if (a.o.p_draft) a.o.p_draft[(int64_t)b * K + lane] = zero ? 0.f : (float)px;
        if (a.o.q_draft) a.o.q_draft[(int64_t)b * K + lane] = zero ? 0.f : (float)qx;
        if (zero && a.o.tv) a.o.tv[(int64_t)b * K + lane] = 0.f;
    }
    if (lane == 0) {
        a.o.accept_len[b] = nn;
        if (a.o.row_status && seq_st) red_or(a.o.row_status + b, seq_st);
    }
    if (fatal) { if (lane == 0) draw_decided(a.fb_count); return; }
    // ---- the draw: position nn (row pair), or the bonus row when every draft was accepted
    const bool pair = nn < L;
    const int du = unit0 + nn;
    const Row rp = pair ? shfl_row(sp, nn) : rb;
    Row rq = shfl_row(sq, pair ? nn : 0);
    if (!pair) { rq.inv_s = 0.0; rq.e = E_EMPTY; rq.st = 0; }
    // The draw's error bound wants sum p^2 + q^2 over the row pair, for which the records carry an upper bound per slice
    // (chunks far below the row's largest logit count next to nothing, and a peaked row gets a bound close to the sum).
    double s2 = 0.0;
    {
        const Rec* base = a.rec + ((int64_t)du * T) * 2;
        for (int i = lane; i < T; i += 32) {
            const Rec r0 = ld_cg(base + 2 * i), r1 = ld_cg(base + 2 * i + 1);
            if (rec_e(r0) > E_EMPTY) { const double f = pow2d(max(rec_e(r0) - rp.e, -500)) * rp.inv_s; s2 += (double)rec_ub(r0) * f * f; }
            if (pair && rec_e(r1) > E_EMPTY) { const double f = pow2d(max(rec_e(r1) - rq.e, -500)) * rq.inv_s; s2 += (double)rec_ub(r1) * f * f; }
        }
    }
    s2 = warp_sum(s2);
    const double bound = draw_bound(s2, (double)a.kappa);
    // the chunk that owns u Z: lanes hold contiguous runs of chunks; the owning lane's run is then spread over the lanes
    const int n4 = T * (CH / 4), per = (n4 + 31) / 32;
    const int i0 = min(lane * per, n4), i1 = min(i0 + per, n4);
    const float* const dm = a.cm + (int64_t)du * T * CH;
    double mine = 0.0;
    if (pair) mine = run_masses(a, S, dm, i0, i1);
    else for (int i = i0; i < i1; ++i) mine += sum4(bonus4(a, S, du, i, rp.e));
    mine *= rp.inv_s;
    double base0, Z, total;
    owner_lane(mine, 0.0, -1.0, &base0, &Z);            // (a target below zero finds no owner: this call is for the total)
    const double Tt = (double)uf * Z;
    int y = -1, cert = 0;
    const int ol = Tt > 0.0 ? owner_lane(mine, 0.0, Tt, &base0, &total) : -1;
    if (ol >= 0) {
        // the run's chunks, 32 at a time: chunk ch = 4 * (ol * per) + lane
        int ch = -1; double cbase = base0;
        for (int g = 0; g < 4 * per && ch < 0; g += 32) {
            const int cc = 4 * (ol * per) + g + lane;
            double m = 0.0;
            if (g + lane < 4 * per && cc < 4 * n4) {
                const float4 v = pair ? ld_relaxed_f4(dm + (cc & ~3)) : bonus4(a, S, du, cc >> 2, rp.e);
                m = (double)((cc & 3) == 0 ? v.x : (cc & 3) == 1 ? v.y : (cc & 3) == 2 ? v.z : v.w) * rp.inv_s;
            }
            double cb, tot;
            const int ow = owner_lane(m, cbase, Tt, &cb, &tot);
            if (ow >= 0) { ch = 4 * (ol * per) + g + ow; cbase = cb; } else cbase = tot;
        }
        if (ch >= 0) {
            const int s = ch / CH, w = ch % CH;
            const int v0 = s * a.slice_vecs + w * CV, nv = max(min(min(a.slice_vecs, R.nvec - s * a.slice_vecs) - w * CV, CV), 0);
            const char* prow = row_ptr(R, b, nn);
            const char* qrow = pair ? row_ptr(R, b, K + 1 + nn) : prow;
            uint4 xp[4], xq[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int vi = j * 32 + lane;
                xp[j] = neg_inf_vec<DT>(); xq[j] = neg_inf_vec<DT>();
                if (vi < nv) {
                    xp[j] = ldg16(prow + (int64_t)(v0 + vi) * 16);
                    if (pair) xq[j] = ldg16(qrow + (int64_t)(v0 + vi) * 16);
                    const int left = V - (v0 + vi) * VEC;
                    if (left < VEC) { mask_tail<DT>(xp[j], left); mask_tail<DT>(xq[j], left); }
                }
            }
            const QExp Ep = chunk_exponent(vecs_max<DT>(xp), ts.hi), Eq = chunk_exponent(vecs_max<DT>(xq), ts.hi);
            const float4 rho = chunk_rho(scale_of(rp, rq), Ep.e, Eq.e);
            const double fp = (Ep.e > E_EMPTY ? pow2d(max(Ep.e - rp.e, -1000)) : 0.0) * rp.inv_s;      // r' (or e) -> probability mass
            // the running sums in front of the vectors (four scans side by side), then the owning lane walks its vector
            double incl[4], dv[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float r[VEC];
                draw_vec<DT>(xp[j], xq[j], pair, ts.hi, Ep, Eq, rho, r);
                dv[j] = (double)sum_fixed<VEC>(r) * fp; incl[j] = dv[j];
            }
#pragma unroll
            for (int o = 1; o < 32; o <<= 1)
#pragma unroll
                for (int j = 0; j < 4; ++j) { const double t2 = shfl_up_d(incl[j], o); if (lane >= o) incl[j] += t2; }
            int at = -1; double C = 0.0, base = cbase;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double lo = base + (incl[j] - dv[j]), hi = base + incl[j];
                if (at < 0 && lo < Tt && Tt <= hi) { at = j; C = lo; }
                base += __shfl_sync(0xffffffffu, incl[j], 31);
            }
            if (at >= 0) {
                float r[VEC];
                draw_vec<DT>(at == 0 ? xp[0] : at == 1 ? xp[1] : at == 2 ? xp[2] : xp[3], at == 0 ? xq[0] : at == 1 ? xq[1] : at == 2 ? xq[2] : xq[3],
                             pair, ts.hi, Ep, Eq, rho, r);
#pragma unroll
                for (int i = 0; i < VEC; ++i) {
                    const double r1 = (double)r[i] * fp, Cn = C + r1;
                    if (y < 0 && r1 > 0.0 && Cn >= Tt) { y = (v0 + at * 32 + lane) * VEC + i; cert = (Tt - C > bound) && (Cn - Tt >= bound); }
                    C = Cn;
                }
            }
        }
    }
    const unsigned found = __ballot_sync(0xffffffffu, y >= 0);
    const bool keep = __popc(found) == 1 && __shfl_sync(0xffffffffu, cert, (__ffs(found) - 1) & 31);
    if (keep) {
        if (y >= 0) { a.o.out_tokens[(int64_t)b * (K + 1) + nn] = y; draw_decided(a.fb_count); }
    } else {
        // listed for the re-draw: its sums and masses are cleared before the record that announces them
        int slot = 0;
        if (lane == 0) slot = draw_listed(a.fb_count);
        slot = __shfl_sync(0xffffffffu, slot, 0);
        for (int i = lane; i < a.nx; i += 32) { a.xsum[(int64_t)slot * a.nx + i] = make_double2(0.0, 0.0); a.xmass[(int64_t)slot * a.nx + i] = 0.0; }
        __threadfence();
        __syncwarp();
        if (lane == 0) st_fb(a.fb_list + slot, b, 2 * nn + (pair ? 1 : 0), rp.e, pair ? rq.e : 0);
    }
    // ---- TV of every position: the sum of its chunks' masses
    if (a.o.tv) for (int k = 0; k < L; ++k) {
        const double z = (k == nn ? Z : warp_sum(run_masses(a, S, a.cm + (int64_t)(unit0 + k) * T * CH, i0, i1)) * __shfl_sync(0xffffffffu, sp.inv_s, k));
        if (lane == 0) a.o.tv[(int64_t)b * K + k] = (float)fmin(fmax(z, 0.0), 1.0);
    }
}

// ------------------------------------------------------------------ fp64 re-draw of the listed sequences
// Warps that have nothing else to do take items (listed sequence, 64 vectors) from a counter.  Everything is
// evaluated in double around the row exponents that the list carries (any common reference cancels in
// p = a / sum a).  An item is: the sums of exponentials of its vectors; once the sums of all the sequence's items are
// there, their residual mass, from the logits still in registers; and the warp that holds item 0 picks the token when all
// masses are there.  Items are taken in order, and whoever holds one is running, so no wait depends on a warp that has
// not started.
struct XRow {
    const char* prow; const char* qrow;
    double c, ep, eq, ip, iq;      // p = exp2(x * c - ep) * ip
    int b, k;
    bool pair;
};
// explicit roundings: a contracted p * ip - q would leave rounding dust when p == q
__device__ __forceinline__ double x_resid(const XRow& d, double pa, double pb, bool two) {
    const double p = __dmul_rn(pa, d.ip);
    if (!two) return p;
    const double df = p - __dmul_rn(pb, d.iq);
    return df > 0.0 ? df : 0.0;
}
template <int DT> __device__ __forceinline__ void x_vec(const uint4& raw, double c, double e, const double* tab, double* t) {
    float f[Elem<DT>::VEC];
    unpack<DT>(raw, f);
#pragma unroll
    for (int i = 0; i < Elem<DT>::VEC; ++i) t[i] = q_exp2(fma((double)f[i], c, -e), tab);
}
// vector `v` of a row; beyond the row or the vocabulary: -inf
template <int DT> __device__ __forceinline__ uint4 x_load(const RowArgs& R, const char* row, int v) {
    uint4 x = neg_inf_vec<DT>();
    if (v < R.nvec) {
        x = ldg16_stream(row + (int64_t)v * 16);
        const int left = R.V - v * Elem<DT>::VEC;
        if (left < Elem<DT>::VEC) mask_tail<DT>(x, left);
    }
    return x;
}
__device__ __forceinline__ double2 ld_sum(const double2* p) {
    unsigned long long w0, w1;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p) : "memory");
    return make_double2(__longlong_as_double((long long)w0), __longlong_as_double((long long)w1));
}
__device__ __forceinline__ double ld_mass(const double* p) { return __longlong_as_double((long long)ld_relaxed64(p)); }

// the token from the items' masses (a plain row has none: its masses are the sums over Sa)
template <int DT>
__device__ __noinline__ void redraw_pick(const StreamArgs& a, Shared& S, XRow d, int slot) {
    constexpr int VEC = Elem<DT>::VEC;
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, nx = a.nx, per = (nx + 31) / 32;
    const int i0 = min(lane * per, nx), i1 = min(i0 + per, nx);
    const double2* xs = a.xsum + (int64_t)slot * nx;
    const double* xm = a.xmass + (int64_t)slot * nx;
    bool two = d.pair, hit;
    auto mass = [&](int i) {
        if (!two) return ld_sum(xs + i).x * d.ip;                      // (all sums have been seen)
        double m = ld_mass(xm + i);
        for (uint32_t t = 0; !there(m) && wait_more(a, S, t, 60); ++t) m = ld_mass(xm + i);
        return m;
    };
    double mine = 0.0;
    for (int i = i0; i < i1; i += 4) {
        double m[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { m[k] = 0.0; if (i + k < i1) m[k] = two ? ld_mass(xm + i + k) : ld_sum(xs + i + k).x * d.ip; }
#pragma unroll
        for (int k = 0; k < 4; ++k) if (i + k < i1) mine += there(m[k]) ? m[k] : mass(i + k);
    }
    double base, Z = warp_sum(mine), tot;
    if (!(Z > 0.0) && two) {
        // residual mass vanished at a rejected position: draw from p of that position
        two = false;
        if (lane == 0 && a.o.row_status) red_or(a.o.row_status + d.b, ST_ZERO_RESID);
        mine = 0.0;
        for (int i = i0; i < i1; ++i) mine += mass(i);
        Z = warp_sum(mine);
    }
    const double t = (double)a.u_final[d.b] * Z;
    const int ol = max(pick_lane(mine, 0.0, t, &base, &tot, &hit), 0);
    int it = ol * per; double cb = base;                               // the lane's items, 32 at a time
    for (int g = 0; g < per; g += 32) {
        const int i = ol * per + g + lane;
        double b0;
        const int src = pick_lane(g + lane < per && i < nx ? mass(i) : 0.0, base, t, &b0, &tot, &hit);
        if (src >= 0) { it = ol * per + g + src; cb = b0; }
        if (hit) break;
        base = tot;
    }
    int y = INT_MAX, last = -1;
#pragma unroll 1
    for (int j = 0; j < XV / 32; ++j) {
        const int v = it * XV + j * 32 + lane;
        double pa[VEC], pb[VEC], vs = 0.0;
        x_vec<DT>(x_load<DT>(R, d.prow, v), d.c, d.ep, S.tab, pa);
        x_vec<DT>(two ? x_load<DT>(R, d.qrow, v) : neg_inf_vec<DT>(), d.c, d.eq, S.tab, pb);
#pragma unroll
        for (int i = 0; i < VEC; ++i) { pa[i] = x_resid(d, pa[i], pb[i], two); vs += pa[i]; }
        double incl = vs;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
        double C = cb + (incl - vs);
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            if (pa[i] > 0.0) { last = v * VEC + i; if (y == INT_MAX && C + pa[i] >= t) y = last; }
            C += pa[i];
        }
        cb += __shfl_sync(0xffffffffu, incl, 31);
    }
    y = __reduce_min_sync(0xffffffffu, y); last = redux_max(last);
    if (lane == 0) a.o.out_tokens[(int64_t)d.b * (R.K + 1) + d.k] = y != INT_MAX ? y : last;
}

template <int DT>
__device__ __noinline__ void redraw_item(const StreamArgs& a, Shared& S, int slot, int it) {
    constexpr int VEC = Elem<DT>::VEC, NJ = XV / 32;
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, nx = a.nx;
    FbRec rec; bool ok = false;
    rec = ld_fb(a.fb_list + slot, &ok);                                // a place in the list is taken before its record is written
    for (uint32_t i = 0; !ok && wait_more(a, S, i, 60); ++i) rec = ld_fb(a.fb_list + slot, &ok);
    if (!__all_sync(0xffffffffu, ok)) return;
    __threadfence();
    XRow d;
    d.b = rec.b1 - 1; d.k = rec.kp >> 1; d.pair = rec.kp & 1;
    d.prow = row_ptr(R, d.b, d.k);
    d.qrow = d.pair ? row_ptr(R, d.b, R.K + 1 + d.k) : d.prow;
    d.c = 1.4426950408889634 / (double)tau_of(R, d.b);
    d.ep = (double)rec.ep; d.eq = (double)rec.eq;
    d.ip = 1.0; d.iq = 0.0;
    uint4 x[NJ], z[NJ];
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        x[j] = x_load<DT>(R, d.prow, it * XV + j * 32 + lane);
        z[j] = d.pair ? x_load<DT>(R, d.qrow, it * XV + j * 32 + lane) : neg_inf_vec<DT>();
    }
    double2* xs = a.xsum + (int64_t)slot * nx;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
        double sa = 0.0, sb = 0.0;
#pragma unroll 1
        for (int j = 0; j < NJ; ++j) {
            double pa[VEC], pb[VEC];
            x_vec<DT>(j ? x[NJ - 1] : x[0], d.c, d.ep, S.tab, pa);
            x_vec<DT>(j ? z[NJ - 1] : z[0], d.c, d.eq, S.tab, pb);
#pragma unroll
            for (int i = 0; i < VEC; ++i) { if (pass == 0) { sa += pa[i]; sb += pb[i]; } else sa += x_resid(d, pa[i], pb[i], true); }
        }
        sa = warp_sum(sa);
        if (pass == 0) {
            sb = warp_sum(sb);
            if (lane == 0) {
                const unsigned long long w0 = (unsigned long long)__double_as_longlong(nonzero_bits(sa)), w1 = (unsigned long long)__double_as_longlong(nonzero_bits(sb));
                asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" :: "l"(xs + it), "l"(w0), "l"(w1) : "memory");
            }
            if (!d.pair && it != 0) return;                            // (a plain row needs no mass pass)
            // exact normalisers: every warp adds the items' sums in the same order
            double Sa = 0.0, Sb = 0.0;
            for (int i = lane; i < nx; i += 128) {
                double2 v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) { v[k] = make_double2(-0.0, -0.0); if (i + 32 * k < nx) v[k] = ld_sum(xs + i + 32 * k); }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    for (uint32_t t = 0; !(there(v[k].x) && there(v[k].y)) && wait_more(a, S, t, 60); ++t) v[k] = ld_sum(xs + i + 32 * k);
                    Sa += v[k].x; Sb += v[k].y;
                }
            }
            Sa = warp_sum(Sa); Sb = warp_sum(Sb);
            d.ip = 1.0 / Sa; d.iq = d.pair ? 1.0 / Sb : 0.0;
            if (!d.pair) break;
        } else if (lane == 0) {
            asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" :: "l"(a.xmass + (int64_t)slot * nx + it), "d"(nonzero_bits(sa)) : "memory");
        }
    }
    if (it == 0) redraw_pick<DT>(a, S, d, slot);
}

// a warp without other work: items until every sequence is decided and the list is worked off
template <int DT>
__device__ __noinline__ void redraw_worker(const StreamArgs& a, Shared& S) {
    const int lane = threadIdx.x & 31;
    if (a.expire == 1) { if (lane == 0) give_up(a, S); return; }         // test hook: the wait for the list has run out already
    bool holds = false;
    unsigned item = 0;
    for (uint32_t i = 0;;) {
        const unsigned long long w = *(volatile unsigned long long*)&S.fbcount;
        const unsigned listed = (unsigned)(w & 0xffffffffull), decided = (unsigned)(w >> 32);
        if (!holds && listed > 0) {
            // (an item that is not listed yet is kept until it is, or the list turns out to end before it)
            if (lane == 0) item = atomicAdd(a.xticket, 1u);
            item = __shfl_sync(0xffffffffu, item, 0);
            holds = true;
        }
        const int slot = holds ? (int)(item / (unsigned)a.nx) : 0;
        if (holds && slot < (int)listed) {
            redraw_item<DT>(a, S, slot, (int)(item - (unsigned)slot * (unsigned)a.nx));
            __syncwarp();
            holds = false; i = 0;
            continue;
        }
        if ((int)decided >= a.r.B || !wait_more(a, S, i++, 150)) return;
    }
}

}  // namespace

template <int DT, bool TVM>
__global__ void __launch_bounds__(ST_THREADS, 1) k_stream(const __grid_constant__ StreamArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    SharedD<DT>& S = *reinterpret_cast<SharedD<DT>*>(smem + Dims<DT>::DATA);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // ---- what the call needs cleared: records, masses, counters, the status words (all warps)
    for (unsigned i = blockIdx.x * ST_THREADS + tid; i < a.zero16; i += gridDim.x * ST_THREADS) reinterpret_cast<uint4*>(a.zero)[i] = make_uint4(0u, 0u, 0u, 0u);
    if (a.o.row_status) for (int i = blockIdx.x * ST_THREADS + tid; i < a.r.B; i += gridDim.x * ST_THREADS) a.o.row_status[i] = 0;
    // The grid meets once: what was cleared is clear for everybody.  Meanwhile the CTA is set up and its first stages are
    // on their way.
    auto grid = cooperative_groups::this_grid();
    auto token = grid.barrier_arrive();
    if (tid == 0) {
        for (int i = 0; i < NSTG; ++i) { mbar_init(&S.full[i], 1); mbar_init(&S.empty[i], CW); }
        for (int i = 0; i < R8; ++i) { mbar_init(&S.pdone[i], CW); mbar_init(&S.stats[i], 1); }
        S.abort = 0; S.failed = 0; S.fbcount = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (!TVM && warp == W_FIN0) { S.tab[lane] = g_pow2_64[lane]; S.tab[lane + 32] = g_pow2_64[lane + 32]; }
    if (warp == 0) tmem_alloc(&S.tmem_base, TCOLS);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    Producer P;
    P.n = 0; P.u = 0; P.st = 0; P.t = blockIdx.x; P.nx.t = -1; P.src = nullptr; P.bytes = 0;
    bool more = true;
    if (warp == W_PROD && lane == 0) {
        if (P.t < a.total) P.nx = fetch_next<TVM>(a, (int)P.t);
        for (int i = 0; i < NSTG && more; ++i) more = produce<DT, TVM, true>(a, S, smem_u32(smem), P);
    }
    grid.barrier_wait(static_cast<cooperative_groups::grid_group::arrival_token&&>(token));
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem0 = S.tmem_base;
    if (warp < CW) {
        consumer<DT, TVM>(a, S, smem_u32(smem), tid);
        if (!TVM) redraw_worker<DT>(a, S);
    } else if (warp == W_PROD) {
        if (lane == 0) {
            while (more) more = produce<DT, TVM, false>(a, S, smem_u32(smem), P);
            produce_stop(a, S, P);
            // the list of the re-draw, for this CTA's warps
            if (!TVM) for (uint32_t i = 0; i < kSpin && !aborted(S); ++i) {
                const unsigned long long w = ld_relaxed64(a.fb_count);
                *(volatile unsigned long long*)&S.fbcount = w;
                if ((int)(w >> 32) >= a.r.B) break;
                __nanosleep(100);
            }
        }
        __syncwarp();
    } else if (warp < W_FIN0) stats_warp<DT>(a, S, warp - W_STAT0);
    else {
        for (int b = (warp - W_FIN0) * (int)gridDim.x + (int)blockIdx.x; b < a.r.B; b += NFIN * (int)gridDim.x) {
            if (TVM) finish_tv(a, S, b); else finish_seq<DT>(a, S, b);
            __syncwarp();
        }
        if (!TVM) redraw_worker<DT>(a, S);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem0, TCOLS);
    // a wait of this CTA gave up: every row's status says so
    if (S.failed && a.o.row_status) for (int i = tid; i < a.r.B; i += ST_THREADS) red_or(a.o.row_status + i, ST_WAIT);
}

// -----------------------------------------------------------------------------
namespace {

template <int DT> constexpr size_t stream_smem() { return (size_t)Dims<DT>::DATA + sizeof(SharedD<DT>); }

template <int DT, bool TVM>
int stream_grid() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64 && cached[dev]) return cached[dev];
    if (cudaFuncSetAttribute(k_stream<DT, TVM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)stream_smem<DT>()) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int per_sm = 0, sms = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_stream<DT, TVM>, ST_THREADS, stream_smem<DT>()) != cudaSuccess) per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    const int n = per_sm >= 1 ? sms : 0;      // the grid must be resident as a whole: one CTA per SM
    if (dev >= 0 && dev < 64) cached[dev] = n;
    return n;
}

}  // namespace

extern cudaEvent_t g_ev_start, g_ev_stop;

bool stream_supported(const RowArgs& a) {
    return make_stream_plan(a.B, a.nvec, a.K + 1).T <= kStreamMaxSlices && a.K <= BEBOP_MAX_K_INT;
}

cudaError_t stream_verify(const RowArgs& a, const Plan& p, const int32_t* draft_tokens, const float* u_accept,
                          const float* u_final, VerifyOut o, char* ws, cudaStream_t stream, bool* launched, bool tv_only,
                          float* s_aux) {
    *launched = false;
    const int grid_max = tv_only ? (a.dt == 0 ? stream_grid<0, true>() : stream_grid<1, true>())
                                 : (a.dt == 0 ? stream_grid<0, false>() : stream_grid<1, false>());
    const int ups = tv_only ? 1 : a.K + 1;
    const StreamPlan sp = make_stream_plan(a.B, a.nvec, ups);
    // the T slices of a unit must be in flight together: T <= grid; and all tasks counted in an int
    if (grid_max < 1 || sp.T > grid_max) return cudaSuccess;
    const int tps = tv_only ? sp.T : a.K * sp.T + (sp.T + 1) / 2;
    const long long total = (long long)a.B * tps;
    if (total > 0x7fff0000LL || (long long)a.B * ups * sp.T > 0x7fff0000LL) return cudaSuccess;
    const int grid = (int)(total < grid_max ? total : grid_max);
    if (grid < sp.T) return cudaSuccess;
    char* w = ws + p.off_pipe;
    StreamArgs fa;
    fa.r = a; fa.draft_tokens = draft_tokens; fa.u_accept = u_accept; fa.u_final = u_final; fa.o = o;
    fa.s_aux = tv_only ? s_aux : nullptr; fa.ups = ups; fa.tps = tps;
    fa.T = sp.T; fa.slice_vecs = sp.slice_vecs; fa.total = (int)total; fa.nx = sp.nx;
    fa.expire = take_expire_wait();
    fa.kappa = draw_kappa();
    fa.zero = w; fa.zero16 = (unsigned)(sp.zero_bytes / 16);
    fa.wait_failed = reinterpret_cast<int*>(w) + 1;
    fa.xticket = reinterpret_cast<unsigned*>(w + kRedrawTicketOffset);
    fa.fb_count = reinterpret_cast<unsigned long long*>(w + kFbCountOffset);
    fa.fb_list = reinterpret_cast<FbRec*>(w + sp.off_fbrec);
    fa.rec = reinterpret_cast<Rec*>(w + sp.off_rec);
    fa.rows = reinterpret_cast<Row*>(w + sp.off_rows);
    fa.cm = reinterpret_cast<float*>(w + sp.off_cm);
    fa.ca = reinterpret_cast<float*>(w + sp.off_ca);
    fa.xsum = reinterpret_cast<double2*>(w + sp.off_xsum);
    fa.xmass = reinterpret_cast<double*>(w + sp.off_xmass);
    if (g_ev_start) cudaEventRecord(g_ev_start, stream);
    // A cooperative launch: the device takes the grid only as a whole, so CTAs of two such grids (two streams) cannot
    // end up holding SMs while each waits for partners that found no room.
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(ST_THREADS); cfg.stream = stream;
    cfg.dynamicSmemBytes = a.dt == 0 ? stream_smem<0>() : stream_smem<1>();
    cfg.attrs = attr; cfg.numAttrs = 1;
    cudaError_t e;
    if (tv_only) e = a.dt == 0 ? cudaLaunchKernelEx(&cfg, k_stream<0, true>, fa) : cudaLaunchKernelEx(&cfg, k_stream<1, true>, fa);
    else e = a.dt == 0 ? cudaLaunchKernelEx(&cfg, k_stream<0, false>, fa) : cudaLaunchKernelEx(&cfg, k_stream<1, false>, fa);
    if (e == cudaErrorCooperativeLaunchTooLarge) { cudaGetLastError(); return cudaSuccess; }     // no room for the whole grid
    if (g_ev_stop) cudaEventRecord(g_ev_stop, stream);
    if (e != cudaSuccess) return e;
    *launched = true;
    return cudaSuccess;
}

}  // namespace bebop
