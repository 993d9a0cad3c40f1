// The fp64 re-draw of the sequences whose fast draw did not clear its error bound (its first kernel also turns
// an expired device-side wait into a status bit), and the hook that times the main kernel.
#include "bebop_chunk.cuh"

namespace bebop {

namespace {

// ------------------------------------------------------------------ fp64 re-draw of the listed sequences
// One small kernel beside the pipelined and the fused kernel, for the few sequences whose fast draw did not clear its
// error bound.  Every row is cut into nx items (a quarter or an eighth of a slice); the items (listed sequence,
// place) are taken from a counter by a grid that fits the device at once.  Everything is evaluated in double
// around the row exponents that phase A left (any common reference cancels in p = a / sum a).  An item is
//   sum    exact normalisers: the sum of exponentials of its vectors of the draw rows, which stay in shared
//          memory; then, once the sums of all items of the sequence are there (a counter per listed sequence),
//   mass   its residual mass; and once all masses are there,
//   token  every CTA finds the item that owns the target, and the one that holds it goes on: the warp's chunk from
//          the masses of its warps, the token from the exponentials.
// What bounds it is a chain, met in full by the last listed sequence, when the main kernel has ended: the list, the
// logits, two exchanges through L2 and the arithmetic of one thread.  So a thread's exponentials run side by side (as a
// choice of doubles, the test for -inf had become a branch around each of them: 170 cycles apiece, one after the
// other), and the token is found where the exponentials are, instead of by the last CTA to finish, which chose with one
// thread and evaluated the chosen chunk again.  A call with re-drawn sequences (2 per cent of them) ends 5 to 8 us earlier:
// 192 sequences of 32,000 bf16 logits, K = 7 ragged, take 84.4 instead of 92.9 us, 256 of 151,936, K = 3, 206 instead of 212.
// A warp per 64 vectors instead of a CTA per item, 300 to 600 items a row, was slower (90 and 239 us): every warp then reads all
// sums and masses, and all of them do the scans, in double, that one CTA's worth of warps does here.
// The kernel is a programmatic dependent of the pipelined kernel that does NOT wait for that grid: its
// CTAs move in as CTAs of the main kernel leave, and work through the list while it still grows (records
// carry a mark; one word counts the listed sequences and the sequences whose draw is decided, which tells the
// end of the list).  The sequences
// listed early are finished before the main kernel ends.
struct RedrawArgs {
    RowArgs r;
    const float* u_final;
    VerifyOut o;
    const unsigned long long* fb_count;   // low half: listed sequences so far; high half: sequences whose draw is decided
    const FbRec* fb_list;    // records, valid once their b1 is non-zero
    int expect;              // sequences that get decided: the list is complete when the high half reaches it
    int* wait_failed;        // set by a device-side wait that gave up
    double2* xsum;           // [B][nx] sums of exponentials (target row, draft row) per item
    double* xmass;           // [B][nx] residual mass per item
    int* xsdone;             // [B] per listed sequence: sum tasks finished
    int* xdone;              // [B] per listed sequence: mass tasks finished
    int expire;              // test hook: the wait for the list gives up at once
    unsigned* xticket;       // [1] next work item
    int nx, item_vecs;       // items per sequence, vectors of an item
};

struct XRow {
    const char* prow; const char* qrow;
    double c, ep, eq, ip, iq;      // p = exp2(x * c - ep) * ip
    int b, k;
    bool pair;
};
// explicit roundings: a contracted p * ip - q would leave rounding dust when p == q
__device__ __forceinline__ double x_resid(const XRow& d, double ea, double eb, bool two) {
    const double p = __dmul_rn(ea, d.ip);
    if (!two) return p;
    const double df = p - __dmul_rn(eb, d.iq);
    return df > 0.0 ? df : 0.0;
}
__device__ __forceinline__ void x_row(const RedrawArgs& a, int slot, XRow* d) {
    const RowArgs& R = a.r;
    bool there;
    const FbRec rec = ld_fb(a.fb_list + slot, &there);          // (x_wait_slot has seen the record valid)
    const int b = rec.b1 - 1, k = rec.kp >> 1;
    d->b = b; d->k = k;
    d->pair = rec.kp & 1;
    d->prow = row_ptr(R, b, k);
    d->qrow = d->pair ? row_ptr(R, b, R.K + 1 + k) : d->prow;
    d->c = 1.4426950408889634 / (double)tau_of(R, b);
    d->ep = (double)rec.ep;
    d->eq = (double)rec.eq;
    d->ip = 1.0; d->iq = 1.0;
}
constexpr int XNU = (kPipeSliceVecs / kRedrawCut + WT - 1) / WT;     // vectors per thread and row in a work item
static_assert(kPipeSliceVecs % (kRedrawCut * 2) == 0 && XNU >= 1 && XNU <= 2, "work items of the fp64 re-draw");

// this thread's vectors of quarter slice s: warp chunk [warp*cw, warp*cw + cw), lanes interleaved
template <int DT>
__device__ __forceinline__ void x_load(const RedrawArgs& a, const XRow& d, int s, float (*fp)[Elem<DT>::VEC],
                                       float (*fq)[Elem<DT>::VEC]) {
    constexpr int VEC = Elem<DT>::VEC;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int qv = a.item_vecs, cw = (qv + WW - 1) / WW;
    const int v0 = s * qv, nv = max(min(qv, a.r.nvec - v0), 0);
#pragma unroll
    for (int u = 0; u < XNU; ++u) {
        const int vl = warp * cw + lane + 32 * u;
        const bool in = lane + 32 * u < cw && vl < nv;
#pragma unroll
        for (int i = 0; i < VEC; ++i) { fp[u][i] = -INFINITY; fq[u][i] = -INFINITY; }
        if (in) {
            load_vec<DT>(d.prow, v0 + vl, a.r.V, fp[u]);
            if (d.pair) load_vec<DT>(d.qrow, v0 + vl, a.r.V, fq[u]);
        }
    }
}

__device__ __forceinline__ unsigned long long x_ld_count(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
// 1: slot is listed and its record is valid; 0: the list is complete and ends before it; -1: a wait gave up
__device__ __forceinline__ int x_wait_slot(const RedrawArgs& a, int slot) {
    if (a.expire) return -1;                             // test hook: this wait's bound has run out already
    uint32_t i = 0;
    for (; i < kSpin; ++i) {
        const unsigned long long w = x_ld_count(a.fb_count);
        if (slot < (int)(w & 0xffffffffull)) break;
        if ((int)(w >> 32) >= a.expect) return 0;
        __nanosleep(256);
    }
    if (i == kSpin) return -1;
    for (i = 0; i < kSpin; ++i) {                       // a place in the list is taken before its record is written
        if (rec_valid(ld_cg(a.fb_list + slot))) return 1;
        __nanosleep(64);
    }
    return -1;
}

template <int DT>
__global__ void __launch_bounds__(WT) k_redraw(const RedrawArgs a) {
    constexpr int VEC = Elem<DT>::VEC;
    __shared__ double shs[2][WW], shm[WW];          // sums and masses of the warps' chunks
    __shared__ double tab[64];
    __shared__ int go;
    __shared__ unsigned item_sh;
    extern __shared__ double xe[];       // [2][XNU * VEC][WT] exponentials of this item's elements (target row, draft row)
    const RowArgs& R = a.r;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid < 64) tab[tid] = g_pow2_64[tid];
    const int K = R.K, XT = a.nx;
    const int qv = a.item_vecs, cw = (qv + WW - 1) / WW;
    const long items_max = (long)R.B * XT;
    __syncthreads();
    // Work items are taken in order from a ticket counter, so the CTAs that are on the device work on the oldest
    // listed sequence; whoever holds an item is running, so the wait for a sequence's other items cannot
    // depend on a CTA that has not started.
    for (;;) {
        if (tid == 0) {
            const unsigned item = atomicAdd(a.xticket, 1u);
            item_sh = item;
            go = item < (unsigned long)items_max ? x_wait_slot(a, (int)(item / (unsigned)XT)) : 0;
        }
        __syncthreads();
        const int g = go;
        const int slot = (int)(item_sh / (unsigned)XT), s = (int)(item_sh - (unsigned)slot * (unsigned)XT);
        __syncthreads();
        if (g <= 0) {                                   // slots come in rising order: nothing behind this one either
            if (g < 0 && tid == 0) atomicExch(a.wait_failed, 1);
            break;
        }
        XRow d;
        x_row(a, slot, &d);
        const int b = d.b;
        const float uf = a.u_final[b];
        // ---- sums of exponentials of this item
        {
            float fp[XNU][VEC], fq[XNU][VEC];
            x_load<DT>(a, d, s, fp, fq);
            double sa = 0.0, sb = 0.0;
#pragma unroll
            for (int u = 0; u < XNU; ++u) {
                if (32 * u >= cw) break;
#pragma unroll
                for (int i = 0; i < VEC; ++i) {
                    const double ea = q_exp2(fma((double)fp[u][i], d.c, -d.ep), tab);
                    sa += ea;
                    // kept for the masses and for the token, which then need neither the rows nor the exponentials again
                    xe[(u * VEC + i) * WT + tid] = ea;
                    if (d.pair) {
                        const double eb = q_exp2(fma((double)fq[u][i], d.c, -d.eq), tab);
                        sb += eb;
                        xe[((XNU + u) * VEC + i) * WT + tid] = eb;
                    }
                }
            }
            sa = warp_sum(sa); sb = warp_sum(sb);
            if (lane == 0) { shs[0][warp] = sa; shs[1][warp] = sb; }
            __syncthreads();
            if (tid == 0) {
                double ta = 0.0, tb = 0.0;
                for (int w = 0; w < WW; ++w) { ta += shs[0][w]; tb += shs[1][w]; }
                a.xsum[(int64_t)b * XT + s] = make_double2(ta, tb);
                __threadfence();
                atomicAdd(a.xsdone + slot, 1);
                // ... and wait (bounded) for the other items of the sequence
                go = spin_ge(a.xsdone + slot, XT) ? 1 : 0;
            }
            __syncthreads();
        }
        bool ok = go != 0;
        // exact normalisers: every warp adds the items' sums in the same order (lane t takes sums t,
        // t + 32, ...; the butterfly leaves the same bits in every lane), so every CTA gets the same value
        double Sa = 0.0, Sb = 0.0;
        if (ok) for (int t = lane; t < XT; t += 32) { const double2 x = __ldcg(a.xsum + (int64_t)b * XT + t); Sa += x.x; Sb += x.y; }
        Sa = warp_sum(Sa); Sb = warp_sum(Sb);
        d.ip = 1.0 / Sa; d.iq = d.pair ? 1.0 / Sb : 0.0;
        if (ok && d.pair) {     // a bonus row needs no mass pass: its masses are sums of exponentials over Sa
            double m = 0.0;
#pragma unroll
            for (int u = 0; u < XNU; ++u) {
                if (32 * u >= cw) break;
#pragma unroll
                for (int i = 0; i < VEC; ++i) m += x_resid(d, xe[(u * VEC + i) * WT + tid], xe[((XNU + u) * VEC + i) * WT + tid], true);
            }
            m = warp_sum(m);
            if (lane == 0) shm[warp] = m;
            __syncthreads();
            if (tid == 0) {
                double t = 0.0;
                for (int w = 0; w < WW; ++w) t += shm[w];
                a.xmass[(int64_t)b * XT + s] = t;
                __threadfence();
                atomicAdd(a.xdone + slot, 1);
                go = spin_ge(a.xdone + slot, XT) ? 1 : 0;
            }
            __syncthreads();
            ok = go != 0;
        }
        if (!ok) {
            if (tid == 0) { atomicExch(a.wait_failed, 1); if (a.o.row_status) atomicOr(a.o.row_status + b, ST_WAIT); }
            __syncthreads();
            continue;
        }
        // ---- the item.  Every warp chooses, from the same numbers in the same order, and the CTA that holds the chosen item
        // goes on.  (The last CTA to finish chose before, by one thread, and evaluated the chosen chunk again.)
        bool two = d.pair, hit;
        const int per = (XT + 31) / 32, t0 = min(lane * per, XT), t1 = min(t0 + per, XT);
        auto mass = [&](int t) { return two ? __ldcg(a.xmass + (int64_t)b * XT + t) : __ldcg(a.xsum + (int64_t)b * XT + t).x * d.ip; };
        double base, tot, t;
        int ol;
        for (;;) {
            double mine = 0.0;
            for (int i = t0; i < t1; ++i) mine += mass(i);
            t = (double)uf * warp_sum(mine);
            ol = pick_lane(mine, 0.0, t, &base, &tot, &hit);
            if (ol >= 0 || !two) break;
            two = false;                                // residual mass vanished at a rejected position: draw from p of that position
        }
        ol = max(ol, 0);
        int qs = ol * per; double cb = base;
        if (per > 1) {
            const int src = pick_lane(lane < per && ol * per + lane < XT ? mass(ol * per + lane) : 0.0, base, t, &cb, &tot, &hit);
            if (src >= 0) qs = ol * per + src;
        }
        if (qs == s) {
            if (tid == 0 && two != d.pair && a.o.row_status) {
                // the main kernel writes this row's status word once, with a plain store: add the bit only when
                // that grid is through (rare, and then a wait of some microseconds at most)
                asm volatile("griddepcontrol.wait;" ::: "memory");
                atomicOr(a.o.row_status + b, ST_ZERO_RESID);
            }
            // ---- the chunk, and the token in it: the first with mass whose running sum reaches the target; by rounding none
            // may: then the last with mass
            double c0;
            const int wsel = max(pick_lane(lane < WW ? (two ? shm[lane] : shs[0][lane] * d.ip) : 0.0, cb, t, &c0, &tot, &hit), 0);
            if (warp == wsel) {
                int y = INT_MAX, last = -1;
#pragma unroll 1
                for (int u = 0; u < XNU; ++u) {
                    const bool in = lane + 32 * u < cw && 32 * u < cw;
                    double r[VEC], vs = 0.0;
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        r[i] = in ? x_resid(d, xe[(u * VEC + i) * WT + tid], xe[((XNU + u) * VEC + i) * WT + tid], two) : 0.0;
                        vs += r[i];
                    }
                    double incl = vs;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
                    double C = c0 + (incl - vs);
                    const int v = s * qv + warp * cw + lane + 32 * u;
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        if (r[i] > 0.0) { last = v * VEC + i; if (y == INT_MAX && C + r[i] >= t) y = last; }
                        C += r[i];
                    }
                    c0 += __shfl_sync(0xffffffffu, incl, 31);
                }
                y = __reduce_min_sync(0xffffffffu, y); last = __reduce_max_sync(0xffffffffu, last);
                if (lane == 0) a.o.out_tokens[(int64_t)b * (K + 1) + d.k] = y != INT_MAX ? y : last;
            }
        }
        __syncthreads();
    }
    // Every CTA waits here for the main grid, whatever the caller asked for: a dependent of a grid that lets its
    // dependents start early has to, or work enqueued behind this kernel (a copy of the results, the next call's
    // clearing of this workspace) would not be ordered behind that grid.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // a wait that gave up, in the main kernel or here: every row's status says so
    if (a.o.row_status && ld_acquire(a.wait_failed) != 0)
        for (int b = blockIdx.x * WT + tid; b < R.B; b += gridDim.x * WT) atomicOr(a.o.row_status + b, ST_WAIT);
}

}  // namespace

cudaEvent_t g_ev_start = nullptr, g_ev_stop = nullptr;
void pipe_set_events(cudaEvent_t start, cudaEvent_t stop) { g_ev_start = start; g_ev_stop = stop; }

namespace {
template <int DT>
constexpr size_t redraw_smem() { return sizeof(double) * 2 * XNU * Elem<DT>::VEC * WT; }
template <int DT>
int redraw_grid() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64 && cached[dev]) return cached[dev];
    int per_sm = 0, sms = 0;
    if (cudaFuncSetAttribute(k_redraw<DT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)redraw_smem<DT>()) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_redraw<DT>, WT, redraw_smem<DT>()) != cudaSuccess) per_sm = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaGetLastError();
    const int n = per_sm * sms;
    if (dev >= 0 && dev < 64) cached[dev] = n;
    return n;
}
}  // namespace

// fp64 re-draw of the listed sequences (usually a few per cent of the batch; the count stays on the device).
// `expect` sequences get their draw decided by the main kernel (0: none, nothing is listed).
cudaError_t redraw_launch(const RowArgs& a, const float* u_final, VerifyOut o, const unsigned long long* fb_count,
                          const FbRec* fb_list, int expect, int* wait_failed, char* w,
                          const PipePlan& wp, cudaStream_t stream, bool expire_list_wait) {
    RedrawArgs ra;
    ra.expire = expire_list_wait ? 1 : 0;
    ra.r = a; ra.u_final = u_final; ra.o = o;
    ra.fb_count = fb_count; ra.fb_list = fb_list; ra.expect = expect;
    ra.wait_failed = wait_failed;
    ra.xsum = reinterpret_cast<double2*>(w + wp.off_xsum);
    ra.xmass = reinterpret_cast<double*>(w + wp.off_xmass);
    ra.xsdone = reinterpret_cast<int*>(w + wp.off_xsdone);
    ra.xdone = reinterpret_cast<int*>(w + wp.off_xdone);
    ra.xticket = reinterpret_cast<unsigned*>(w + kRedrawTicketOffset);
    const int cut = redraw_cut(wp.T);
    ra.nx = cut * wp.T; ra.item_vecs = wp.slice_vecs / cut;
    // CTAs of this grid wait for one another (the sums of a sequence come from nx of them), so
    // the grid is at most what fits the device at once; a CTA takes work items from a counter.
    const int cap = a.dt == 0 ? redraw_grid<0>() : redraw_grid<1>();
    if (cap < 1) return cudaErrorLaunchOutOfResources;
    const long items_max = (long)a.B * ra.nx;
    const int grid = (int)(items_max < cap ? items_max : cap);
    // scheduled as soon as the main kernel lets go of SMs; it does not wait for that grid as a whole
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(WT); cfg.stream = stream;
    cfg.dynamicSmemBytes = a.dt == 0 ? redraw_smem<0>() : redraw_smem<1>();
    cfg.attrs = attr; cfg.numAttrs = 1;
    return a.dt == 0 ? cudaLaunchKernelEx(&cfg, k_redraw<0>, ra) : cudaLaunchKernelEx(&cfg, k_redraw<1>, ra);
}

}  // namespace bebop
