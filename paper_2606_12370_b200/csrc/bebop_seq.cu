// Sequence kernel: bebop_verify, bebop_tv and the greedy mode with one thread-block cluster per sequence (row pair), for
// the calls whose time is latency: few sequences, or rows short enough that a sequence's logits fit the shared memory of
// the cluster (up to sixteen CTAs, 3.5 MB).
//
// A CTA of the cluster holds its slice of every row of the sequence in shared memory (bulk copies, all started at
// once, one barrier per row) and works on chunks of 128 16-byte vectors, a warp each:
//   pass 1  the chunk's reference exponent E (an integer) and sum of e = 2^(x c - E); the rows' sums are merged over
//           the warps, then -- every CTA sends its own to all others through distributed shared memory -- over the cluster;
//   scan    the accept scan (Algorithm 3), by every CTA for itself, on the same numbers;
//   pass 2  the residuals max(0, p - q) of the row pairs that TV or the draw needs, from the logits in shared memory;
//           the CTAs exchange their masses; the CTA that owns the target u Z of the inverse CDF finds the token and keeps it if
//           the crossing clears the error bound of the fp32 prefix sums;
//   re-draw when it does not, the cluster evaluates the draw rows again in double, from shared memory, at once.
// So a call is one launch with three exchanges of about a microsecond inside a cluster: no workspace to clear, no
// grid-wide meeting, no kernel behind it.  What other sequences do does not matter, so nothing can wait on a CTA that
// has not started (a cluster is placed as a whole).
//
// What bounds it: latency.  A call of four sequences of 1,024 fp32 logits (K = 3) takes 7.5 to 7.9 us (28 through the pipelined
// kernel with its clearing and its re-draw kernel); its parts, timed inside the kernel, are in that order of size: start 1.8, pass 1
// 0.5, the exchange 1.5, scan 0.4, pass 2 1.3, exchange 0.9, draw 2.  A re-draw adds 5 to 10 (24 when its exponentials were spread over the chunks' warps only).  One sequence of 151,936 bf16
// logits, sixteen CTAs of 133 KB: 16 us (32), of which the exponentials of the two passes take 7.
#include "bebop_chunk.cuh"

namespace bebop {

namespace {

constexpr int QV = 4;                         // vectors per lane of a chunk
constexpr int QCV = 32 * QV;                  // vectors per chunk
constexpr int kSeqThreads = 512;              // threads per CTA, at most
constexpr int kSeqMaxCluster = 16;
constexpr uint32_t kQSpin = 1u << 24;

// offsets of a CTA's tables behind the logits in shared memory (bytes)
struct SeqPlan {
    int C, sv, nch, rows;                     // CTAs per sequence, vectors per row slice, chunks per slice, rows held
    int o_psum, o_pexp, o_cm, o_ca, o_rec, o_stat, o_rho, o_rmass, o_raux, o_rx, o_x, o_bar, bytes;
};

struct SeqArgs {
    RowArgs r;
    const int32_t* draft_tokens;
    const float* u_accept;
    const float* u_final;
    VerifyOut o;
    float* s_aux;
    SeqPlan p;
    int expire;                               // test hook: the wait for the rows counts as run out
    float kappa;
};

struct __align__(16) QRec { double s, ub; int e, bad; double pad; };    // a row's sum around 2^e, bound of its sum of squares
struct __align__(16) QStat { double inv_s, ub; int e, st; double pad; };

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ bool mbar_wait(unsigned long long* b) {
    const uint32_t addr = smem_u32(b);
    for (uint32_t i = 0; i < kQSpin; ++i) if (mbar_try(addr, 0)) return true;
    return false;
}
// log2(e) / tau, finite whatever tau: 0 * c is 0
__device__ __forceinline__ float seq_scale(float tau) { return fminf(temp_scale(tau).hi, 3e38f); }
// vector `vi` of a row slice of nv vectors; what lies beyond the slice or the vocabulary reads as -inf
template <int DT>
__device__ __forceinline__ uint4 slice_vec(const unsigned char* row, int vi, int nv, int v0, int V) {
    constexpr int VEC = Elem<DT>::VEC;
    uint4 x = neg_inf_vec<DT>();
    if (vi < nv) {
        x = *reinterpret_cast<const uint4*>(row + (size_t)vi * 16);
        const int left = V - (v0 + vi) * VEC;
        if (left < VEC) mask_tail<DT>(x, left);
    }
    return x;
}
// the lane's vectors of chunk c (interleaved: j * 32 + lane); `full`: the chunk lies inside the slice and the vocabulary
template <int DT>
__device__ __forceinline__ void chunk_vecs(const unsigned char* row, int c, bool full, int nv, int v0, int V, uint4* x) {
    const int vi = c * QCV + (threadIdx.x & 31);
    if (full) {
#pragma unroll
        for (int j = 0; j < QV; ++j) x[j] = *reinterpret_cast<const uint4*>(row + (size_t)(vi + j * 32) * 16);
    } else {
#pragma unroll
        for (int j = 0; j < QV; ++j) x[j] = slice_vec<DT>(row, vi + j * 32, nv, v0, V);
    }
}
// r' = max(0, e_p - rho e_q) = (p - q) S_p, rho = S_p / S_q as two floats (equal rows give rho = 1 and 0 exactly; the
// large product first, so that the small one decides the sign where q is close to p); as e_p <= 1, saturating to [0, 1] is
// taking the maximum with 0
template <int DT>
__device__ __forceinline__ void resid_vec(const float* ep, const float* eq, float2 rho, float* r) {
#pragma unroll
    for (int i = 0; i < Elem<DT>::VEC; ++i) r[i] = fma_sat(-rho.y, eq[i], fmaf(-rho.x, eq[i], ep[i]));
}
// What the threads of a CTA share besides the tables of the plan.
struct QShared {
    double tab[64];                           // 2^(j/64), for the re-draw
    double target, base;                      // of the draw
    int nn, status, owner, keep, failed;      // stop position; status bits; rank that owns the target; the token was kept
};

// the rows' records of all CTAs (rrec[rank][row], sent by their owners) merged: the same bits in every CTA
__device__ __forceinline__ void merge_cluster(const SeqArgs& a, const QRec* rrec, QStat* stat, int rows) {
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int i = threadIdx.x >> 5; i < rows; i += nw) {
        QRec r; r.s = 0.0; r.ub = 0.0; r.e = E_EMPTY; r.bad = 0;
        if (lane < a.p.C) r = rrec[lane * a.p.rows + i];
        const int Em = redux_max(r.e), bad = __reduce_or_sync(0xffffffffu, r.bad);
        const double f = r.e > E_EMPTY ? pow2d(max(r.e - Em, -1000)) : 0.0;
        const double s = warp_sum(r.s * f), ub = warp_sum(r.ub * f * f);
        if (lane == 0) {
            QStat x;
            x.st = (bad & 2) ? ST_WAIT : ((bad & 1) || !(s == s)) ? ST_NONFINITE : Em == E_EMPTY ? ST_EMPTY : far_exponent(Em) ? ST_FAR : 0;
            x.inv_s = !x.st && s > 0.0 ? 1.0 / s : 0.0; x.e = Em; x.ub = ub * x.inv_s * x.inv_s; x.pad = 0.0;
            stat[i] = x;
        }
    }
}

// Rows marked ST_FAR are moved into the range of the reference exponents: every logit becomes x - m, m the row's maximum, in the
// shared memory of all CTAs.  That is exact wherever it matters: a logit within a factor of two of m differs from it by a
// number of the same type, and any other lies at least |m| / 2 below, 2^(-2e6) of the row's largest weight.  The
// softmax does not change, and pass 1 runs again.  Ordinary calls only pay for the test of the statuses, which they make
// anyway (one sequence of 151,936 bf16 logits 15.8 -> 16.1 us, the other calls measured alike); a call, never made, to a
// function that evaluates such a sequence in double, or a flag of its own, cost 0.2 to 0.3 us in all of them.
template <int DT>
__device__ __forceinline__ void move_far_rows(const SeqArgs& a, unsigned char* smem, const QStat* stat, int* rmax, int rows, int nv, int v0, int rank) {
    constexpr int VEC = Elem<DT>::VEC;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    cluster_sync();                                         // (every CTA has merged: the rows' records may be written again)
#pragma unroll 1
    for (int i = warp; i < rows; i += nw) {
        if (stat[i].st != ST_FAR) continue;
        const unsigned char* const row = smem + (size_t)i * a.p.sv * 16;
        float m = -INFINITY;
#pragma unroll 1
        for (int v = lane; v < nv; v += 32) m = fmaxf(m, vec_max<DT>(slice_vec<DT>(row, v, nv, v0, a.r.V)));
        const int om = redux_max(f2ord(m));
        if (lane < a.p.C) st_remote(at_rank(rmax + rank * a.p.rows + i, lane), om);
    }
    cluster_sync();
#pragma unroll 1
    for (int i = warp; i < rows; i += nw) {
        if (stat[i].st != ST_FAR) continue;
        uint4* const row = reinterpret_cast<uint4*>(smem + (size_t)i * a.p.sv * 16);
        const float m = ord2f(redux_max(lane < a.p.C ? rmax[lane * a.p.rows + i] : INT_MIN));
#pragma unroll 1
        for (int v = lane; v < nv; v += 32) {
            float f[VEC];
            unpack<DT>(row[v], f);
#pragma unroll
            for (int j = 0; j < VEC; ++j) f[j] -= m;
            row[v] = pack<DT>(f);
        }
    }
}

// The accept scan by one warp: lane k owns draft position k.  Leaves the stop position and the status; rank 0 writes
// accept_len, the accepted tokens, p, q and the status.
__device__ __forceinline__ void accept_scan(const SeqArgs& a, QShared& S, const QStat* stat, int b, int L, float tau, int tk, float u,
                                            float zpx, float zqx, bool write) {
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, K = R.K;
    const float c = seq_scale(tau);
    const bool active = lane < L, tok_ok = tk >= 0 && tk < R.V;
    int seq_st = tau_ok(tau) ? 0 : ST_BAD_TEMP;
    QStat sp, sq;
    sp.inv_s = 0.0; sp.e = 0; sp.st = 0; sq = sp;
    if (active) { sp = stat[2 * lane]; sq = stat[2 * lane + 1]; }
    const QStat sb = stat[2 * L];
    const int wait = __reduce_or_sync(0xffffffffu, (sp.st | sq.st | sb.st) & ST_WAIT);
    if (!seq_st && __ballot_sync(0xffffffffu, active && !tok_ok)) seq_st = ST_BAD_TOKEN;
    // the first bad row pair decides the status; rows after it do not count
    const int rs = active ? (sp.st | sq.st) : 0;
    const unsigned badrows = __ballot_sync(0xffffffffu, rs != 0);
    const int first_bad = badrows ? __ffs(badrows) - 1 : 32;
    const int rs_first = __shfl_sync(0xffffffffu, rs, first_bad & 31);
    if (!seq_st && badrows) seq_st = rs_first;
    double px = 0.0, qx = 0.0;
    bool acc = false;
    if (active && !(seq_st & ST_STOP) && lane < first_bad) {
        const double cd = (double)c;
        px = exp2((double)zpx * cd - (double)sp.e) * sp.inv_s;
        qx = exp2((double)zqx * cd - (double)sq.e) * sq.inv_s;
        acc = (double)u * qx < px;
    }
    const unsigned rej = __ballot_sync(0xffffffffu, active && !acc);
    const int n = rej ? __ffs(rej) - 1 : L;
    if (!(seq_st & ST_STOP) && n == L) seq_st |= sb.st;               // bonus row, counted only now
    if (wait) seq_st = ST_WAIT;
    const bool fatal = (seq_st & (ST_STOP | ST_WAIT)) != 0;
    const int nn = fatal ? 0 : n;
    if (write) {
        for (int q = lane; q <= K; q += 32)
            if (fatal || q != nn) a.o.out_tokens[(int64_t)b * (K + 1) + q] = q < nn ? tk : -1;       // (q < nn <= 32: q == lane)
        if (lane < K) {
            const bool zero = fatal || lane >= L;
            if (a.o.p_draft) a.o.p_draft[(int64_t)b * K + lane] = zero ? 0.f : (float)px;
            if (a.o.q_draft) a.o.q_draft[(int64_t)b * K + lane] = zero ? 0.f : (float)qx;
            if (zero && a.o.tv) a.o.tv[(int64_t)b * K + lane] = 0.f;
        }
        if (lane == 0) { a.o.accept_len[b] = nn; if (a.o.row_status) a.o.row_status[b] = seq_st; }
    }
    if (lane == 0) { S.nn = nn; S.status = seq_st; }
}

// The fp32 draw, by one warp of the CTA that owns the target: chunk from the chunk masses `cm` (units of 1 / inv), token
// from the chunk's vectors.  True: the token is certified and written.
template <int DT>
__device__ __forceinline__ bool fast_draw(const SeqArgs& a, const unsigned char* prow, const unsigned char* qrow, bool pair, const QStat& sp, const QStat& sq,
                                          float2 rho, float c, const double* cm, double base, double Tt, int nv, int v0, int32_t* out) {
    constexpr int VEC = Elem<DT>::VEC;
    const int lane = threadIdx.x & 31;
    const double bound = draw_bound(sp.ub + (pair ? sq.ub : 0.0), (double)a.kappa);
    int ch = -1;
    for (int g = 0; g < a.p.nch && ch < 0; g += 32) {
        double b0, tot;
        const int ow = owner_lane(g + lane < a.p.nch ? cm[g + lane] * sp.inv_s : 0.0, base, Tt, &b0, &tot);
        if (ow >= 0) { ch = g + ow; base = b0; } else base = tot;
    }
    if (ch < 0) return false;
    // the chunk's vectors, and the running sums in front of them (four scans side by side)
    float r[QV][VEC];
    double incl[QV], dv[QV];
#pragma unroll
    for (int j = 0; j < QV; ++j) {
        float ep[VEC];
        exp_vec<DT>(slice_vec<DT>(prow, ch * QCV + j * 32 + lane, nv, v0, a.r.V), c, (float)sp.e, ep);
        if (pair) {
            float eq[VEC];
            exp_vec<DT>(slice_vec<DT>(qrow, ch * QCV + j * 32 + lane, nv, v0, a.r.V), c, (float)sq.e, eq);
            resid_vec<DT>(ep, eq, rho, r[j]);
        } else {
#pragma unroll
            for (int i = 0; i < VEC; ++i) r[j][i] = ep[i];
        }
        dv[j] = (double)sum_fixed<VEC>(r[j]) * sp.inv_s;
        incl[j] = dv[j];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int j = 0; j < QV; ++j) { const double t2 = shfl_up_d(incl[j], o); if (lane >= o) incl[j] += t2; }
    int y = -1, cert = 0, at = -1;
    double C = 0.0;
#pragma unroll
    for (int j = 0; j < QV; ++j) {
        const double lo = base + (incl[j] - dv[j]), hi = base + incl[j];
        if (at < 0 && lo < Tt && Tt <= hi) { at = j; C = lo; }
        base += __shfl_sync(0xffffffffu, incl[j], 31);
    }
    if (at >= 0) {
#pragma unroll
        for (int i = 0; i < VEC; ++i) {
            const float ri = at == 0 ? r[0][i] : at == 1 ? r[1][i] : at == 2 ? r[2][i] : r[3][i];
            const double r1 = (double)ri * sp.inv_s, Cn = C + r1;
            if (y < 0 && r1 > 0.0 && Cn >= Tt) { y = (v0 + ch * QCV + at * 32 + lane) * VEC + i; cert = (Tt - C > bound) && (Cn - Tt >= bound); }
            C = Cn;
        }
    }
    const unsigned found = __ballot_sync(0xffffffffu, y >= 0);
    const bool keep = __popc(found) == 1 && __shfl_sync(0xffffffffu, cert, (__ffs(found) - 1) & 31);
    if (keep && y >= 0) *out = y;
    return keep;
}

// The draw rows evaluated again in double, by the whole cluster: exact normalisers, residual masses, the token.  Any
// common reference cancels in p = a / sum a, so the rows' exponents serve.  A warp takes 32 vectors at a time (the work is
// small, and this spreads it over the warps); one piece of code serves both passes (it runs once, from a cold
// instruction cache).
template <int DT>
__device__ __noinline__ void redraw(const SeqArgs& a, QShared& S, unsigned char* tables, const unsigned char* prow, const unsigned char* qrow,
                                    bool pair, const QStat& sp, const QStat& sq, float tau, int nv, int v0, int rank, int b, double u, int32_t* out) {
    constexpr int VEC = Elem<DT>::VEC;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5, n4 = (nv + 31) >> 5;
    double* const xa = reinterpret_cast<double*>(tables + a.p.o_x);           // per 32 vectors: sums of the target row
    double* const xb = xa + QV * a.p.nch;                                     // ... of the draft row, later residual masses
    double* const rx = reinterpret_cast<double*>(tables + a.p.o_rx);          // [C][4]: sums of both rows, mass; by rank
    const double cd = 1.4426950408889634 / (double)tau;
    double ip = 1.0, iq = 0.0;
    // the exponentials of vector vi of both rows
    auto eval = [&](int vi, bool two, double* pa, double* pb) {
#pragma unroll 1
        for (int w = 0; w < 2; ++w) {
            float f[VEC];
            double t[VEC];
            unpack<DT>(w == 0 || two ? slice_vec<DT>(w ? qrow : prow, vi, nv, v0, a.r.V) : neg_inf_vec<DT>(), f);
            const double e = w ? (double)sq.e : (double)sp.e;
#pragma unroll
            for (int i = 0; i < VEC; ++i) t[i] = q_exp2(fma((double)f[i], cd, -e), S.tab);
            if (w == 0) {
#pragma unroll
                for (int i = 0; i < VEC; ++i) pa[i] = t[i];
            } else {
#pragma unroll
                for (int i = 0; i < VEC; ++i) pb[i] = t[i];
            }
        }
    };
    // explicit roundings: a contracted p * ip - q would leave rounding dust when p == q
    auto resid = [&](double pa, double pb, bool two) {
        const double p = __dmul_rn(pa, ip), d = p - __dmul_rn(pb, iq);
        return two ? (d > 0.0 ? d : 0.0) : p;
    };
#pragma unroll 1
    for (int pass = 0; pass < (pair ? 2 : 1); ++pass) {
        for (int q = warp; q < n4; q += nw) {
            double pa[VEC], pb[VEC], sa = 0.0, sb = 0.0;
            eval(q * 32 + lane, pair, pa, pb);
#pragma unroll
            for (int i = 0; i < VEC; ++i) {
                if (pass == 0) { sa += pa[i]; sb += pb[i]; } else sb += resid(pa[i], pb[i], true);
            }
            sa = warp_sum(sa); sb = warp_sum(sb);
            if (lane == 0) { if (pass == 0) xa[q] = sa; xb[q] = sb; }
        }
        __syncthreads();
        if (warp == 0) {
            double sa = 0.0, sb = 0.0;
            for (int q = lane; q < n4; q += 32) { sa += xa[q]; sb += xb[q]; }
            sa = warp_sum(sa); sb = warp_sum(sb);
            if (lane < a.p.C) {
                const uint32_t d = at_rank(rx + 4 * rank, lane);
                if (pass == 0) { st_remote(d, sa); st_remote(d + 8, sb); } else st_remote(d + 16, sb);
            }
        }
        cluster_sync();
        if (pass == 0) {
            double sa = lane < a.p.C ? rx[4 * lane] : 0.0, sb = lane < a.p.C ? rx[4 * lane + 1] : 0.0;
            sa = warp_sum(sa); sb = warp_sum(sb);
            ip = 1.0 / sa; iq = pair ? 1.0 / sb : 0.0;
        }
    }
    if (warp != 0) return;
    bool two = pair, hit;
    double m = lane < a.p.C ? (two ? rx[4 * lane + 2] : rx[4 * lane] * ip) : 0.0;
    double base, Z = warp_sum(m), tot;
    if (!(Z > 0.0) && two) {
        // residual mass vanished at a rejected position: draw from p of that position
        two = false;
        if (rank == 0 && lane == 0 && a.o.row_status) a.o.row_status[b] = S.status | ST_ZERO_RESID;
        m = lane < a.p.C ? rx[4 * lane] * ip : 0.0;
        Z = warp_sum(m);
    }
    const double t = u * Z;
    if (pick_lane(m, 0.0, t, &base, &tot, &hit) != rank) return;
    // the 32 vectors, then the token, by the same rule
    int q0 = 0; double cb = base;
    for (int g = 0; g < n4; g += 32) {
        const double v = g + lane < n4 ? (two ? xb[g + lane] : xa[g + lane] * ip) : 0.0;
        double b0;
        const int src = pick_lane(v, base, t, &b0, &tot, &hit);
        if (src >= 0) { q0 = g + src; cb = b0; }
        if (hit) break;
        base = tot;
    }
    double pa[VEC], pb[VEC], vs = 0.0;
    eval(q0 * 32 + lane, two, pa, pb);
#pragma unroll
    for (int i = 0; i < VEC; ++i) { pa[i] = resid(pa[i], pb[i], two); vs += pa[i]; }
    double incl = vs;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
    double C = cb + (incl - vs);
    int y = INT_MAX, last = -1;
    const int tok0 = (v0 + q0 * 32 + lane) * VEC;
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
        if (pa[i] > 0.0) { last = tok0 + i; if (y == INT_MAX && C + pa[i] >= t) y = last; }
        C += pa[i];
    }
    y = __reduce_min_sync(0xffffffffu, y); last = redux_max(last);
    if (lane == 0) *out = y != INT_MAX ? y : last;
}

}  // namespace

template <int DT, bool TVM>
__global__ void __launch_bounds__(kSeqThreads, 2) k_seq(const __grid_constant__ SeqArgs a) {
    constexpr int VEC = Elem<DT>::VEC;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ QShared S;
    const RowArgs& R = a.r;
    const int C = a.p.C, sv = a.p.sv, nch = a.p.nch;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
    const int rank = (int)cluster_rank(), b = (int)(blockIdx.x / (unsigned)C);
    unsigned char* const tables = smem;                     // (the plan's offsets count from the start; the logits come first)
    double* const psum = reinterpret_cast<double*>(tables + a.p.o_psum);
    int* const pexp = reinterpret_cast<int*>(tables + a.p.o_pexp);
    double* const cm = reinterpret_cast<double*>(tables + a.p.o_cm);
    double* const ca = reinterpret_cast<double*>(tables + a.p.o_ca);
    QRec* const rrec = reinterpret_cast<QRec*>(tables + a.p.o_rec);
    QStat* const stat = reinterpret_cast<QStat*>(tables + a.p.o_stat);
    float2* const rho = reinterpret_cast<float2*>(tables + a.p.o_rho);
    double* const rmass = reinterpret_cast<double*>(tables + a.p.o_rmass);
    double* const raux = reinterpret_cast<double*>(tables + a.p.o_raux);
    unsigned long long* const bar = reinterpret_cast<unsigned long long*>(tables + a.p.o_bar);
    auto row_of = [&](int i) { return smem + (size_t)i * sv * 16; };          // row 2k: target k, 2k + 1: draft k, 2L: bonus
    cluster_arrive();                                       // (waited for before the first store into another CTA)
    if (warp == 0) {
        for (int i = lane; i < a.p.rows; i += 32) mbar_init(&bar[i], 1);
        if (lane == 0) S.failed = a.expire;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (!TVM && warp == nw - 2) { S.tab[lane] = g_pow2_64[lane]; S.tab[lane + 32] = g_pow2_64[lane + 32]; }
    __syncthreads();
    // The launch of this grid overlaps the end of the one before it in the stream (programmatic dependent launch): nothing
    // of the caller's memory is touched until that grid is through.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int L = TVM ? 1 : len_of(R, b);
    const float tau = tau_of(R, b), c = seq_scale(tau);
    const int rows = TVM ? 2 : 2 * L + 1;
    const int v0 = rank * sv, nv = max(min(sv, R.nvec - v0), 0);
    const int nfull = v0 + nv == R.nvec && R.V % VEC != 0 ? nv - 1 : nv;      // vectors that hold no token beyond the vocabulary
    if (warp == 0 && nv > 0)
        for (int i = lane; i < rows; i += 32) {
            const int r = (i & 1) ? R.K + 1 + (i >> 1) : (i >> 1);
            mbar_arrive_expect(&bar[i], (uint32_t)nv * 16u);
            bulk_load(smem_u32(row_of(i)), row_ptr(R, b, r) + (int64_t)v0 * 16, (uint32_t)nv * 16u, &bar[i]);
        }
    // the last warp runs the accept scan: lane k owns draft position k, whose token, uniform and logits are asked for now
    const int aw = nw - 1;
    int tk = 0; float u = 0.f, zpx = 0.f, zqx = 0.f;
    if (!TVM && warp == aw && lane < L) {
        tk = a.draft_tokens[(int64_t)b * R.K + lane]; u = a.u_accept[(int64_t)b * R.K + lane];
        if (tk >= 0 && tk < R.V) { zpx = load_one<DT>(row_ptr(R, b, lane), tk); zqx = load_one<DT>(row_ptr(R, b, R.K + 1 + lane), tk); }
    }
    const float uf = !TVM && warp == 0 ? a.u_final[b] : 0.f;
    // ---- pass 1: a warp per (row, chunk).  (Once more when the statuses say that rows lie beyond its range; what stands between
    // here and pass 2 writes the same places again then.)
    for (bool moved = false;; moved = true) {
        for (int it = warp; it < rows * nch; it += nw) {
            const int i = it / nch, ch = it - i * nch;
            double s = 0.0;
            int e = E_EMPTY;
            if (ch * QCV < nv) {
                if (!mbar_wait(&bar[i])) S.failed = 1;
                uint4 x[QV];
                chunk_vecs<DT>(row_of(i), ch, (ch + 1) * QCV <= nfull, nv, v0, R.V, x);
                const QExp E = chunk_exponent(max_nan(max_nan(vec_max<DT>(x[0]), vec_max<DT>(x[1])), max_nan(vec_max<DT>(x[2]), vec_max<DT>(x[3]))), c);
                float sum = 0.f;
#pragma unroll
                for (int j = 0; j < QV; ++j) { float f[VEC]; exp_vec<DT>(x[j], c, E.ef, f); sum += sum_fixed<VEC>(f); }
                e = E.e;
                s = e == E_BAD ? 0.0 : warp_sum_fixed(sum);
            }
            if (lane == 0) { psum[it] = s; pexp[it] = e; }
        }
        if (!moved) cluster_wait();                         // every CTA of the cluster has started
        __syncthreads();
        // ---- the CTA's sum of every row, sent to all CTAs
        for (int i = warp; i < rows; i += nw) {
            int em = E_EMPTY;
            for (int k = lane; k < nch; k += 32) em = max(em, pexp[i * nch + k]);
            em = redux_max(em);
            const int bad = em == E_BAD;                        // (what the row's sum is then does not matter)
            double s = 0.0, ub = 0.0;
            for (int k = lane; k < nch; k += 32) {
                const int e = pexp[i * nch + k];
                const double f = e > E_EMPTY && e != E_BAD ? pow2d(max(e - em, -500)) : 0.0;
                s += psum[i * nch + k] * f; ub += psum[i * nch + k] * f * f;        // (e <= 1: a chunk's sum of e^2 is at most its sum of e)
            }
            s = warp_sum(s); ub = warp_sum(ub);
            if (lane < C) {
                const uint32_t d = at_rank(rrec + rank * a.p.rows + i, lane);
                st_remote(d, s); st_remote(d + 8, ub); st_remote(d + 16, em); st_remote(d + 20, bad | (S.failed ? 2 : 0));
            }
        }
        cluster_sync();
        merge_cluster(a, rrec, stat, rows);
        __syncthreads();
        // ---- the accept scan (bebop_tv: the pair's status)
        if (TVM) {
            if (tid == 0) { const int w = (stat[0].st | stat[1].st) & ST_WAIT; S.status = w ? w : !tau_ok(tau) ? ST_BAD_TEMP : (stat[0].st | stat[1].st); S.nn = -1; }
        } else if (warp == aw) accept_scan(a, S, stat, b, L, tau, tk, u, zpx, zqx, rank == 0);
        if (warp == 0) for (int k = lane; k < L; k += 32) {
            const double r = stat[2 * k].inv_s > 0.0 ? stat[2 * k + 1].inv_s / stat[2 * k].inv_s : 0.0;
            rho[k] = make_float2((float)r, (float)(r - (double)(float)r));
        }
        __syncthreads();
        if (__builtin_expect(!(S.status & (ST_STOP | ST_WAIT)), 1)) break;
        if (moved || !(S.status & ST_FAR)) {                // (the same in every CTA: nothing more is sent)
            if (TVM && rank == 0 && tid == 0) {
                a.o.tv[b] = 0.f;
                if (a.s_aux) a.s_aux[b] = 0.f;
                if (a.o.row_status) a.o.row_status[b] = S.status;
            }
            return;
        }
        int* const rmax = reinterpret_cast<int*>(rmass);    // [C][rows held]
        move_far_rows<DT>(a, smem, stat, rmax, rows, nv, v0, rank);
        if (!TVM && warp == aw && lane < L)
            for (int w = 0; w < 2; ++w) if (stat[2 * lane + w].st == ST_FAR) {
                int om = INT_MIN;
                for (int q = 0; q < C; ++q) om = max(om, rmax[q * a.p.rows + 2 * lane + w]);
                if (w) zqx -= ord2f(om); else zpx -= ord2f(om);
            }
        __syncthreads();
    }
    const int nn = S.nn;
    // ---- pass 2: a warp per (row pair, chunk); without a TV output only the pair a token is drawn from
    const bool all = TVM || a.o.tv;
    const int k0 = all ? 0 : nn, pairs = all ? L : (nn < L ? 1 : 0);
    for (int it = warp; it < pairs * nch; it += nw) {
        const int k = k0 + it / nch, ch = it % nch;
        const float ep = (float)stat[2 * k].e, eq = (float)stat[2 * k + 1].e;
        const float2 rh = rho[k];
        double z = 0.0; float sx = 0.f;
        if (ch * QCV < nv) {
            uint4 xp[QV], xq[QV];
            chunk_vecs<DT>(row_of(2 * k), ch, (ch + 1) * QCV <= nfull, nv, v0, R.V, xp);
            chunk_vecs<DT>(row_of(2 * k + 1), ch, (ch + 1) * QCV <= nfull, nv, v0, R.V, xq);
#pragma unroll
            for (int j = 0; j < QV; ++j) {
                float p[VEC], q[VEC], r[VEC];
                exp_vec<DT>(xp[j], c, ep, p);
                exp_vec<DT>(xq[j], c, eq, q);
                if (TVM) {
                    // q <= p: e_p - rho e_q >= 0; the sum S of Eq. tv_grad goes with the residuals
#pragma unroll
                    for (int i = 0; i < VEC; ++i) {
                        const float d = fmaf(-rh.y, q[i], fmaf(-rh.x, q[i], p[i]));
                        r[i] = fmaxf(d, 0.f);
                        sx += d >= 0.f ? q[i] : 0.f;
                    }
                } else resid_vec<DT>(p, q, rh, r);
                z += (double)sum_fixed<VEC>(r);
            }
        }
        z = warp_sum(z);
        if (TVM) { const double x = warp_sum((double)sx); if (lane == 0) ca[ch] = x; }
        if (lane == 0) cm[k * nch + ch] = z;
    }
    // (bonus row: the chunks' sums around the row's exponent)
    if (!TVM && nn == L && warp == nw - 1) for (int k = lane; k < nch; k += 32) {
        const int e = pexp[2 * L * nch + k];
        cm[L * nch + k] = e > E_EMPTY ? psum[2 * L * nch + k] * pow2d(max(e - stat[2 * L].e, -1000)) : 0.0;
    }
    __syncthreads();
    // ---- the CTA's masses, sent to all CTAs
    for (int i = warp; i < pairs + (!TVM && nn == L ? 1 : 0); i += nw) {
        const int k = i < pairs ? k0 + i : L;
        double z = 0.0, x = 0.0;
        for (int g = lane; g < nch; g += 32) { z += cm[k * nch + g]; if (TVM) x += ca[g]; }
        z = warp_sum(z);
        if (TVM) x = warp_sum(x);
        if (lane < C) {
            st_remote(at_rank(rmass + rank * (R.K + 1) + k, lane), z);
            if (TVM) st_remote(at_rank(raux + rank, lane), x);
        }
    }
    cluster_sync();
    if (rank == 0 && all && tid < L) {
        double z = 0.0;
        for (int r = 0; r < C; ++r) z += rmass[r * (R.K + 1) + tid];
        a.o.tv[(int64_t)b * R.K + tid] = (float)fmin(fmax(z * stat[2 * tid].inv_s, 0.0), 1.0);
        if (TVM) {
            if (a.s_aux) { double x = 0.0; for (int r = 0; r < C; ++r) x += raux[r]; a.s_aux[b] = (float)(x * stat[1].inv_s); }
            if (a.o.row_status) a.o.row_status[b] = 0;
        }
    }
    if (TVM) return;
    // ---- the draw: position nn (row pair), or the bonus row when every draft was accepted
    const bool pair = nn < L;
    const QStat sp = stat[2 * nn], sq = stat[pair ? 2 * nn + 1 : 2 * nn];
    const unsigned char* const prow = row_of(2 * nn);
    const unsigned char* const qrow = row_of(pair ? 2 * nn + 1 : 2 * nn);
    int32_t* const out = a.o.out_tokens + (int64_t)b * (R.K + 1) + nn;
    if (warp == 0) {
        const double m = lane < C ? rmass[lane * (R.K + 1) + nn] * sp.inv_s : 0.0;
        double incl = m;
#pragma unroll
        for (int o = 1; o < kSeqMaxCluster; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
        double lo = shfl_up_d(incl, 1);
        if (lane == 0) lo = 0.0;
        const double Tt = (double)uf * __shfl_sync(0xffffffffu, incl, kSeqMaxCluster - 1);
        const unsigned owners = __ballot_sync(0xffffffffu, lane < C && Tt > lo && Tt <= incl);
        const int own = Tt > 0.0 && owners ? __ffs(owners) - 1 : -1;
        const double base = __shfl_sync(0xffffffffu, lo, own & 31);
        if (own == rank) {
            const int keep = fast_draw<DT>(a, prow, qrow, pair, sp, sq, pair ? rho[nn] : make_float2(0.f, 0.f), c, cm + nn * nch, base, Tt, nv, v0, out) ? 1 : 0;
            if (lane < C) st_remote(at_rank(&S.keep, lane), keep);
        }
        if (lane == 0) { S.owner = own; S.target = (double)uf; }
    }
    cluster_sync();
    if (S.owner >= 0 && S.keep) return;
    redraw<DT>(a, S, tables, prow, qrow, pair, sp, sq, tau, nv, v0, rank, b, S.target, out);
}

// ------------------------------------------------------------------ greedy mode
// A cluster per sequence: its warps take the maximum and the lowest index that has it over pieces of the L + 1 target
// rows, straight from global memory; the CTAs send theirs to rank 0, which runs the argmax match.
struct __align__(8) QMax { int ord, idx; };           // order-preserving integer of the maximum (NaN on top); lowest index
struct SeqGreedyArgs {
    RowArgs r;
    const int32_t* draft_tokens;
    int32_t* accept_len;
    int32_t* out_tokens;
    int32_t* row_status;
    int C, sv, nch;                           // CTAs per sequence, vectors per row slice, pieces per slice
};
constexpr int QGV = 8;                        // vectors per lane of a piece, all asked for at once
__device__ __forceinline__ QMax better(QMax x, QMax y) { return (y.ord > x.ord || (y.ord == x.ord && y.idx < x.idx)) ? y : x; }

template <int DT>
__global__ void __launch_bounds__(kSeqThreads, 2) k_seq_greedy(const __grid_constant__ SeqGreedyArgs a) {
    constexpr int VEC = Elem<DT>::VEC;
    extern __shared__ __align__(128) unsigned char smem[];
    const RowArgs& R = a.r;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int rank = (int)cluster_rank(), b = (int)(blockIdx.x / (unsigned)a.C), K = R.K;
    QMax* const part = reinterpret_cast<QMax*>(smem);                       // [K + 1][nch]
    QMax* const all = part + (K + 1) * a.nch;                               // [K + 1][C] by rank
    cluster_arrive();
    asm volatile("griddepcontrol.wait;" ::: "memory");       // (as in k_seq)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int L = len_of(R, b), rows = L + 1;
    const int v0 = rank * a.sv, nv = max(min(a.sv, R.nvec - v0), 0);
    for (int it = warp; it < rows * a.nch; it += nw) {
        const int i = it / a.nch, ch = it - i * a.nch;
        const char* row = row_ptr(R, b, i);
        uint4 x[QGV];
#pragma unroll
        for (int j = 0; j < QGV; ++j) {
            const int vi = (ch * QGV + j) * 32 + lane;
            x[j] = neg_inf_vec<DT>();
            if (vi < nv) x[j] = ldg16_stream(row + (int64_t)(v0 + vi) * 16);
        }
        float m = -INFINITY;
#pragma unroll
        for (int j = 0; j < QGV; ++j) {
            const int left = R.V - (v0 + (ch * QGV + j) * 32 + lane) * VEC;
            if (left < VEC) mask_tail<DT>(x[j], left);
            m = max_nan(m, vec_max<DT>(x[j]));
        }
        if (!(m < INFINITY)) m = __int_as_float(0x7fc00000);      // NaN or +inf poisons the row
        m += 0.f;                                                 // -0 becomes +0: the integer order must not tell them apart
        int idx = INT_MAX;
#pragma unroll
        for (int j = QGV - 1; j >= 0; --j) {
            float f[VEC];
            unpack<DT>(x[j], f);
#pragma unroll
            for (int q = VEC - 1; q >= 0; --q) if (f[q] == m) idx = (v0 + (ch * QGV + j) * 32 + lane) * VEC + q;
        }
        QMax w;
        const int om = f2ord(m);
        w.ord = redux_max(om);
        w.idx = __reduce_min_sync(0xffffffffu, om == w.ord ? idx : INT_MAX);
        if (lane == 0) part[it] = w;
    }
    cluster_wait();                                         // every CTA of the cluster has started
    __syncthreads();
    for (int i = warp; i < rows; i += nw) {
        QMax w; w.ord = f2ord(-INFINITY); w.idx = INT_MAX;
        for (int k = lane; k < a.nch; k += 32) w = better(w, part[i * a.nch + k]);
        const int om = redux_max(w.ord), im = __reduce_min_sync(0xffffffffu, w.ord == om ? w.idx : INT_MAX);
        if (lane == 0) { const uint32_t d = at_rank(all + i * a.C + rank, 0); st_remote(d, om); st_remote(d + 4, im); }
    }
    cluster_sync();
    if (rank != 0 || warp != 0) return;
    int st = 0, g = -1, g_bonus = -1;
    const int tok = lane < L ? a.draft_tokens[(int64_t)b * K + lane] : -1;
    if (lane < L && (tok < 0 || tok >= R.V)) st |= ST_BAD_TOKEN;
    for (int round = 0; round < 2; ++round) {               // lanes 0..L merge the target rows 0..L (two rounds when L = 32)
        const int k = round * 32 + lane;
        if (k <= L) {
            QMax w = all[k * a.C];
            for (int r = 1; r < a.C; ++r) w = better(w, all[k * a.C + r]);
            const float m = ord2f(w.ord);
            if (m != m) st |= ST_NONFINITE; else if (m == -INFINITY) st |= ST_EMPTY;
            if (round == 0) g = w.idx; else g_bonus = w.idx;
        }
    }
    st = __reduce_or_sync(0xffffffffu, st);
    const bool fatal = (st & ST_FATAL) != 0;
    const unsigned mis = __ballot_sync(0xffffffffu, lane < L && tok != g);
    const int n = fatal ? 0 : mis ? __ffs(mis) - 1 : L;
    const int y = fatal ? -1 : n < 32 ? __shfl_sync(0xffffffffu, g, n & 31) : __shfl_sync(0xffffffffu, g_bonus, 0);
    if (lane <= K) a.out_tokens[(int64_t)b * (K + 1) + lane] = lane < n ? tok : lane == n ? y : -1;
    if (K == 32 && lane == 0) a.out_tokens[(int64_t)b * 33 + 32] = n == 32 ? y : -1;
    if (lane == 0) { a.accept_len[b] = n; if (a.row_status) a.row_status[b] = st; }
}

// -----------------------------------------------------------------------------
namespace {

constexpr int kSeqSmem = 232448 - 1024;       // dynamic shared memory of a CTA, at most (the rest: QShared)

SeqPlan seq_plan(int rows, int K, int nvec, int C) {
    SeqPlan p;
    p.C = C; p.rows = rows;
    p.sv = (nvec + C - 1) / C;
    p.nch = (p.sv + QCV - 1) / QCV;
    const long long data = (long long)rows * p.sv * 16;
    if (data > kSeqSmem) { p.bytes = INT_MAX; return p; }
    int o = (int)data;
    const auto take = [&](int bytes) { const int at = o; o += (bytes + 15) & ~15; return at; };
    p.o_psum = take(8 * rows * p.nch);
    p.o_pexp = take(4 * rows * p.nch);
    p.o_cm = take(8 * (K + 1) * p.nch);
    p.o_ca = take(8 * p.nch);
    p.o_rec = take((int)sizeof(QRec) * C * rows);
    p.o_stat = take((int)sizeof(QStat) * rows);
    p.o_rho = take(8 * (K + 1));
    p.o_rmass = take(8 * C * (K + 1));
    p.o_raux = take(8 * C);
    p.o_rx = take(32 * C);
    p.o_x = take(8 * 2 * QV * p.nch);
    p.o_bar = take(8 * rows);
    p.bytes = o <= kSeqSmem ? o : INT_MAX;
    return p;
}
// the smallest cluster that holds a sequence (0: none does)
int seq_cluster(int rows, int K, int nvec) {
    for (int C = 1; C <= kSeqMaxCluster; ++C) if (seq_plan(rows, K, nvec, C).bytes != INT_MAX) return C;
    return 0;
}
int sm_count() {
    static int cached[64] = {0};
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev >= 0 && dev < 64 && cached[dev]) return cached[dev];
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { cudaGetLastError(); return 0; }
    if (dev >= 0 && dev < 64) cached[dev] = n;
    return n;
}
template <auto kernel> bool seq_ready() {
    static bool done[64] = {false};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    if (dev >= 0 && dev < 64 && done[dev]) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSeqSmem) != cudaSuccess ||
        cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) { cudaGetLastError(); return false; }
    if (dev >= 0 && dev < 64) done[dev] = true;
    return true;
}
// The cluster size for a call: a share per CTA that lets two CTAs run on an SM (one's exchanges then overlap the other's
// arithmetic, and a re-draw is spread over more SMs: 300 sequences of 12,000 bf16 logits, K = 3, take 51 instead of 60 us,
// 48 of 32,000 20 instead of 33), as far as sixteen CTAs go; and more while SMs would idle and the CTAs have work.
constexpr int kSeqShare = 112000;
// How many clusters of C CTAs the device holds at a time, one CTA per SM or two (asked once per device; 0: not known).
// A cluster stays inside one of the chip's GPCs, so large ones leave SMs over.  The answers on a B200, one CTA per SM / two: eight CTAs
// 15 / 33, nine 15 / 30, ten 11 / 26, eleven and twelve 7 / 21, thirteen 7 / 17, fourteen to sixteen 7 / 14.
int seq_resident(int C, bool two) {
    static int cached[64][2][kSeqMaxCluster + 1] = {{{0}}};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) { cudaGetLastError(); return 0; }
    int& n = cached[dev][two][C];
    if (n) return n > 0 ? n : 0;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C); cfg.blockDim = dim3(kSeqThreads); cfg.dynamicSmemBytes = two ? kSeqShare : kSeqSmem;
    cfg.attrs = attr; cfg.numAttrs = 1;
    int got = 0;
    if (!seq_ready<k_seq<1, false>>() || cudaOccupancyMaxActiveClusters(&got, k_seq<1, false>, &cfg) != cudaSuccess) { cudaGetLastError(); got = 0; }
    n = got > 0 ? got : -1;
    return got > 0 ? got : 0;
}
int seq_cluster_for(int B, int rows, int K, int nvec, int dt) {
    const int least = seq_cluster(rows, K, nvec);
    int C = least;
    if (!C) return 0;
    while (C < kSeqMaxCluster && seq_plan(rows, K, nvec, C).bytes > kSeqShare) ++C;
    const int sms = sm_count();
    if (C > 8 && B > 1) {
        // Clusters beyond the portable size leave SMs unused: the size whose waves are done first, a wave taken as 6 us and
        // 0.08 us per KB of bf16 logits in a CTA's share, half of that for fp32 (half as much again where two CTAs share an SM).  24 ragged fp32 sequences of 49,999
        // logits, K = 5: ten CTAs each instead of sixteen, 44 -> 33 us; 8 of 151,936 bf16, K = 3, 32 -> 20.
        double best = 1e30;
        for (int c = least; c <= kSeqMaxCluster; ++c) {
            const int bytes = seq_plan(rows, K, nvec, c).bytes;
            if (bytes == INT_MAX) continue;
            const bool two = bytes <= kSeqShare;
            const int n = seq_resident(c, two);
            if (!n) continue;
            const double t = (double)((B + n - 1) / n) * (6.0 + (two ? 0.12e-3 : 0.08e-3) * (dt == 0 ? 0.5 : 1.0) * bytes);
            if (t < best) { best = t; C = c; }
        }
        return C;
    }
    while (C < kSeqMaxCluster && (long long)B * (C + 1) <= sms && (long long)rows * nvec > (long long)C * 2048) ++C;
    return C;
}
template <typename K, typename A> cudaError_t seq_launch(K kernel, const A& args, int B, int C, int threads, int smem, cudaStream_t stream) {
    cudaLaunchAttribute attr[2];
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)B * (unsigned)C); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
    // a cluster of one CTA is launched as a plain grid, which starts 0.4 to 0.9 us sooner (four sequences of 1,024 fp32 logits
    // 8.8 -> 7.9 us a call); the kernel's cluster instructions then mean the CTA itself
    cfg.attrs = C == 1 ? attr + 1 : attr; cfg.numAttrs = C == 1 ? 1 : 2;
    return cudaLaunchKernelEx(&cfg, kernel, args);
}

}  // namespace

extern cudaEvent_t g_ev_start, g_ev_stop;

bool seq_supported(const RowArgs& a, bool tv_only) {
    return (long long)a.B * kSeqMaxCluster < 0x7fffffffLL && seq_cluster(tv_only ? 2 : 2 * a.K + 1, a.K, a.nvec) > 0;
}

// Where the lines lie, measured against the other kernels (B200, us per call, bf16 and K = 3 unless said).  A sequence that
// one or two CTAs hold: faster at any batch (1,024 sequences of 1,024 logits 28 against 94, 3,000 of 4,096 123 against 184,
// 1,024 of 12,000 121 against 134; fp32 logits fill the CTAs with half the work: 700 of 4,096 51 against 67, but 3,000 of them
// slower; bebop_tv 3,000 pairs of 12,000 67 against 88, but 1,024 of 32,000, two CTAs each, 65 against 58).  Larger clusters
// leave SMs unused (seven clusters of sixteen run at a time) and run in waves without overlap: faster while the call
// is a few waves (128 of 32,000 50 against 57; 24 fp32 ragged ones of 49,999, K = 5, 36
// against 54; one of 151,936 16 against 32), slower beyond (300 of 32,000 103 against 85; 16 of 151,936 44.6 against 42); with nine CTAs, of which fifteen to thirty
// clusters run at a time, somewhat longer (32 of 65,536 31.7 against 39, 40 35.8 against 37.7; the line stands there, though on inputs
// that re-draw in the other kernels it could lie higher: 48 40.5 against 49.7).
bool seq_preferred(const RowArgs& a, bool tv_only) {
    const int rows = tv_only ? 2 : 2 * a.K + 1;
    int C = seq_cluster(rows, a.K, a.nvec);
    if (!C) return false;
    while (C < kSeqMaxCluster && seq_plan(rows, a.K, a.nvec, C).bytes > kSeqShare) ++C;
    const double logits = (double)a.B * rows * a.V;
    if (C == 1) return true;
    // (Longer rows would be faster streamed from about 20 million logits on -- 250 of 16,000 57.0 against 41.4, 128 of 32,000 50.6 against
    // 44.7, 1,000 of 8,000 90 against 70 -- but stay here, where rows far from zero are right.  Beyond the line the stream: 2,000 of 8,000 118
    // against 158, 2,000 of 5,000, K = 8, 192 against 252, 1,000 of 2,000 fp32, K = 8, 80 against 86; of rows below 400 vectors a unit is too
    // little between two exchanges.)
    if (C == 2 && !tv_only && a.nvec < 400) return true;
    if (C == 2) return logits <= (tv_only || a.dt == 0 ? 30e6 : 100e6);
    if (C <= 8) return logits <= (tv_only ? 15e6 : 30e6);
    if (C == 9 && !tv_only) return logits <= 20e6;
    return logits <= (tv_only ? 6e6 : 14e6);
}
// Faster than the sweep of the pipelined kernel and its two companions up to about 100 MB of target logits (7 against 11 us
// for the smallest calls, 20.5 against 23.4 at 67 MB), slower beyond 150 MB.
bool seq_greedy_preferred(const RowArgs& a) { return (double)a.B * (a.K + 1) * a.nvec * 16 <= 100e6; }

cudaError_t seq_verify(const RowArgs& a, const int32_t* draft_tokens, const float* u_accept, const float* u_final, VerifyOut o,
                       cudaStream_t stream, bool* launched, bool tv_only, float* s_aux) {
    *launched = false;
    const int rows = tv_only ? 2 : 2 * a.K + 1;
    const int C = seq_cluster_for(a.B, rows, a.K, a.nvec, a.dt);
    if (!C) return cudaSuccess;
    SeqArgs sa;
    sa.r = a; sa.draft_tokens = draft_tokens; sa.u_accept = u_accept; sa.u_final = u_final; sa.o = o; sa.s_aux = tv_only ? s_aux : nullptr;
    sa.p = seq_plan(rows, a.K, a.nvec, C);
    sa.kappa = draw_kappa();
    const bool ready = tv_only ? (a.dt == 0 ? seq_ready<k_seq<0, true>>() : seq_ready<k_seq<1, true>>())
                               : (a.dt == 0 ? seq_ready<k_seq<0, false>>() : seq_ready<k_seq<1, false>>());
    if (!ready) return cudaSuccess;
    sa.expire = take_expire_wait() ? 2 : 0;
    const int threads = (long long)a.B * C > 2LL * sm_count() && sa.p.bytes < 75000 ? 256 : 512;
    if (g_ev_start) cudaEventRecord(g_ev_start, stream);
    cudaError_t e;
    if (tv_only) e = a.dt == 0 ? seq_launch(k_seq<0, true>, sa, a.B, C, threads, sa.p.bytes, stream) : seq_launch(k_seq<1, true>, sa, a.B, C, threads, sa.p.bytes, stream);
    else e = a.dt == 0 ? seq_launch(k_seq<0, false>, sa, a.B, C, threads, sa.p.bytes, stream) : seq_launch(k_seq<1, false>, sa, a.B, C, threads, sa.p.bytes, stream);
    if (g_ev_stop) cudaEventRecord(g_ev_stop, stream);
    if (e != cudaSuccess) { cudaGetLastError(); return cudaSuccess; }        // (no room for such a cluster: the caller takes another kernel)
    *launched = true;
    return cudaSuccess;
}

cudaError_t seq_greedy(const RowArgs& a, const int32_t* draft_tokens, int32_t* accept_len, int32_t* out_tokens, int32_t* row_status,
                       cudaStream_t stream, bool* launched) {
    *launched = false;
    const int sms = sm_count();
    int C = 1;
    while (C < kSeqMaxCluster && (long long)a.B * (C + 1) <= 2 * sms && (long long)(a.K + 1) * a.nvec > (long long)C * 2048) ++C;
    SeqGreedyArgs ga;
    ga.r = a; ga.draft_tokens = draft_tokens; ga.accept_len = accept_len; ga.out_tokens = out_tokens; ga.row_status = row_status;
    ga.C = C; ga.sv = (a.nvec + C - 1) / C; ga.nch = (ga.sv + 32 * QGV - 1) / (32 * QGV);
    const long long smem = 8LL * (a.K + 1) * (ga.nch + C);
    if (smem > 48 * 1024 || (long long)a.B * C > 0x7fffffffLL) return cudaSuccess;
    if (!(a.dt == 0 ? seq_ready<k_seq_greedy<0>>() : seq_ready<k_seq_greedy<1>>())) return cudaSuccess;
    const cudaError_t e = a.dt == 0 ? seq_launch(k_seq_greedy<0>, ga, a.B, C, 512, (int)smem, stream) : seq_launch(k_seq_greedy<1>, ga, a.B, C, 512, (int)smem, stream);
    if (e != cudaSuccess) { cudaGetLastError(); return cudaSuccess; }
    *launched = true;
    return cudaSuccess;
}

}  // namespace bebop
