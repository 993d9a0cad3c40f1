// What the stream, the pipelined, the re-draw and the sequence kernel share: barriers and bulk copies, the exponentials of a
// chunk around an integer exponent, fixed-point warp sums, owners of a target among the lanes of a warp, 2^t in double.
#pragma once
#include "bebop_pipe.cuh"

namespace bebop {

namespace {

constexpr int E_BAD = 0x3fffffff;             // in place of an exponent: a NaN or +inf was seen

// ------------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long* b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect(unsigned long long* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(smem_u32(b)) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(addr), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, unsigned long long* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// ---- a cluster: its barrier, the shared memory of its other CTAs
// (aligned: all lanes of a warp execute them together, which nothing but a __syncwarp() makes a warp do that has split before)
__device__ __forceinline__ void cluster_arrive() { __syncwarp(); asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { __syncwarp(); asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
__device__ __forceinline__ uint32_t cluster_rank() { uint32_t r; asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
// the address of `p` (this CTA's shared memory) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t at_rank(const void* p, int rank) {
    uint32_t a; asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank)); return a;
}
__device__ __forceinline__ void st_remote(uint32_t a, double v) {
    asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, int v) {
    asm volatile("st.shared::cluster.s32 [%0], %1;" :: "r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ int redux_add(int v) { int r; asm volatile("redux.sync.add.s32 %0, %1, 0xffffffff;" : "=r"(r) : "r"(v)); return r; }
__device__ __forceinline__ float fma_sat(float a, float b, float c) {      // min(max(a b + c, 0), 1), rounded once
    float d; asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c)); return d;
}

// ------------------------------------------------------------------ chunks
// Reference exponent of a chunk from its maximum m: ceil(m c), found by adding 1.5 * 2^23 with rounding upwards, so
// that every e = 2^(x c - E) is at most 1.  The sum of a finite m with |m c| < 2^22 is a float in [2^23, 2^24), whose bit
// pattern grows with its value: the warp's maximum is one integer reduction, and NaN, +inf, -inf in every lane
// and huge logits show as a result outside that range.
constexpr float kMagic = 12582912.f;                  // 1.5 * 2^23
constexpr int kMagicBits = 0x4B400000;
struct QExp { int e; float ef; };
__device__ __forceinline__ QExp chunk_exponent(float m, float c) {
    const int yi = redux_max(__float_as_int(__fmaf_ru(m, c, kMagic)));
    QExp x;
    if (yi >= 0x4B000000 && yi <= 0x4B7FFFFF) { x.e = yi - kMagicBits; x.ef = __int_as_float(yi) - kMagic; return x; }
    const float mw = ord2f(redux_max(f2ord(m)));      // (NaN sorts above +inf)
    x.ef = 0.f; x.e = E_EMPTY;
    if (!(mw < INFINITY)) { x.e = E_BAD; return x; }
    if (mw == -INFINITY) return x;                    // around 0 the chunk's -inf logits give e = 0
    const float y = __fadd_ru(fminf(fmaxf(mw * c, -(float)kFarExp), (float)kFarExp), kMagic);      // (at either end: far_exponent)
    x.ef = y - kMagic; x.e = __float_as_int(y) - kMagicBits;
    return x;
}
// Sum over a warp of a number in [0, 32], as an integer in units of 2^-40, in two words: every lane's number is split
// into a multiple of 2^-17 and the rest, both read off the bits of a float addition, and the integers are added by one
// instruction each.  The sum does not depend on an order and is exact to 2^-40.
constexpr unsigned kSumBits0 = 0x42800000u, kSumBits1 = 0x37400000u;      // 64.0 (ulp 2^-17) and 1.5 * 2^-17 (ulp 2^-40)
constexpr int kNoSum0 = (int)(32u * kSumBits0), kNoSum1 = (int)(32u * kSumBits1);      // what a warp of zeros adds up to
__device__ __forceinline__ int2 warp_sum_words(float x) {
    const float y = __fadd_rn(x, 64.f), r = __fsub_rn(x, __fsub_rn(y, 64.f)), z = __fadd_rn(r, __int_as_float((int)kSumBits1));
    return make_int2(redux_add(__float_as_int(y)), redux_add(__float_as_int(z)));
}
// (an integer as a double by its bits: a conversion waits behind the exponentials of the other warps, whose unit it shares)
__device__ __forceinline__ double int_value(int v) { return __hiloint2double(0x43300000, (int)((unsigned)v ^ 0x80000000u)) - 4503601774854144.0; }      // 2^52 + 2^31
__device__ __forceinline__ double word_value(int2 w) {                 // exact
    return fma(int_value((int)((unsigned)w.x - (unsigned)kNoSum0)), 7.62939453125e-06, int_value((int)((unsigned)w.y - (unsigned)kNoSum1)) * 9.094947017729282e-13);      // 2^-17, 2^-40
}
__device__ __forceinline__ double warp_sum_fixed(float x) { return word_value(warp_sum_words(x)); }
// the largest logit of a lane's N vectors (NaN if there is one); bf16: packed maxima, unpacked once
template <int DT, int N> __device__ __forceinline__ float vecs_max(const uint4* v) {
    if (DT == 1) {
        uint32_t m[N];
#pragma unroll
        for (int j = 0; j < N; ++j) m[j] = max_nan_bf16x2(max_nan_bf16x2(v[j].x, v[j].y), max_nan_bf16x2(v[j].z, v[j].w));
#pragma unroll
        for (int j = 1; j < N; ++j) m[0] = max_nan_bf16x2(m[0], m[j]);
        return max_nan(__uint_as_float(m[0] << 16), __uint_as_float(m[0] & 0xffff0000u));
    }
    float m = vec_max<DT>(v[0]);
#pragma unroll
    for (int j = 1; j < N; ++j) m = max_nan(m, vec_max<DT>(v[j]));
    return m;
}
// the exponentials of one vector around exponent Ef, two at a time
template <int DT>
__device__ __forceinline__ void exp_vec(const uint4& raw, float c, float Ef, float* e) {
    constexpr int VEC = Elem<DT>::VEC;
    float f[VEC];
    unpack<DT>(raw, f);
    const float2 c2 = make_float2(c, c), m2 = make_float2(-Ef, -Ef);
#pragma unroll
    for (int i = 0; i < VEC; i += 2) {
        const float2 t = __ffma2_rn(make_float2(f[i], f[i + 1]), c2, m2);
        e[i] = ex2f(t.x);
        e[i + 1] = ex2f(t.y);
    }
}
// sum of N floats, two at a time (one fixed order)
template <int N> __device__ __forceinline__ float sum_fixed(const float* e) {
    float2 acc = make_float2(e[0], e[1]);
#pragma unroll
    for (int i = 2; i < N; i += 2) acc = __fadd2_rn(acc, make_float2(e[i], e[i + 1]));
    return acc.x + acc.y;
}
// The warp's sum of the lanes' N vector sums, at most 32 times 2^SC a lane, as warp_sum_words of its 2^-SC, without further rounding
// above 2^-38: each is split into a multiple of 2^-17 and the rest, two at a time.  The masses a token is drawn from are such sums:
// added up in fp32, a lane's 64 tokens put a prefix of a flat row (151,936 logits N(0, 1), 20 rows on the host) off by up to 1.8 times
// 2^-22 sqrt(sum p^2), the unit of the draw's bound; eight of them, a vector's, by 0.8.
template <int N, int SC> __device__ __forceinline__ int2 vector_sum_words(const float* v) {
    constexpr unsigned kBase = kSumBits0 + ((unsigned)SC << 23), kRest = 0x38C00000u + ((unsigned)SC << 23);          // 64 and 1.5 * 2^-14 (ulp 2^-37), times 2^SC
    const float b = __int_as_float((int)kBase);
    const float2 base = make_float2(b, b), below = make_float2(-b, -b), minus = make_float2(-1.f, -1.f);
    unsigned hi = kSumBits0 - (unsigned)N * kBase;
    float2 r = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < N; i += 2) {
        const float2 x = make_float2(v[i], v[i + 1]), y = __fadd2_rn(x, base), z = __ffma2_rn(__fadd2_rn(y, below), minus, x);
        hi += (unsigned)__float_as_int(y.x) + (unsigned)__float_as_int(y.y);
        r = i == 0 ? z : __fadd2_rn(r, z);
    }
    const int lo = redux_add(__float_as_int(__fadd_rn(r.x + r.y, __int_as_float((int)kRest))));
    return make_int2(redux_add((int)hi), (int)(((unsigned)lo - 32u * kRest) * 8u + (unsigned)kNoSum1));
}
// Pass 1 of a chunk of Q vectors a lane around exponent Ef: half its sum of exponentials, in words, and the lane's sum.  EXACT (a
// sequence's rows, the bonus row among them): the vectors' sums are added exactly; bebop_tv, which draws nothing, adds a lane's
// tokens in fp32 (256 x 151,936 178.1 us with fp32 sums for both, 181.4 with exact ones; as a branch for bonus rows alone 181.8 and up).
template <int DT, int Q, bool EXACT>
__device__ __forceinline__ int2 chunk_sum(const uint4* x, float c, float Ef, float* sum) {
    constexpr int VEC = Elem<DT>::VEC;
    if constexpr (EXACT) {
        float v[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float e[VEC];
            exp_vec<DT>(x[i], c, Ef, e);
            v[i] = sum_fixed<VEC>(e);
        }
        float2 t = make_float2(v[0], v[1]);
#pragma unroll
        for (int i = 2; i < Q; i += 2) t = __fadd2_rn(t, make_float2(v[i], v[i + 1]));
        *sum = t.x + t.y;
        return vector_sum_words<Q, 1>(v);
    } else {
        float2 s0 = make_float2(0.f, 0.f), s1 = s0;
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float e[VEC];
            exp_vec<DT>(x[i], c, Ef, e);
#pragma unroll
            for (int q = 0; q < VEC; q += 4) { s0 = __fadd2_rn(s0, make_float2(e[q], e[q + 1])); s1 = __fadd2_rn(s1, make_float2(e[q + 2], e[q + 3])); }
        }
        *sum = (s0.x + s0.y) + (s1.x + s1.y);
        return warp_sum_words(0.5f * *sum);
    }
}
// Owner of the target t of an inverse CDF among values that the lanes hold in order (`below` lies before lane 0): its
// lane (-1: none), the running sum before it in *base, the total in *total.
__device__ __forceinline__ int owner_lane(double v, double below, double t, double* base, double* total) {
    const int lane = threadIdx.x & 31;
    double incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
    double excl = shfl_up_d(incl, 1);
    if (lane == 0) excl = 0.0;
    *total = below + __shfl_sync(0xffffffffu, incl, 31);
    const double lo = below + excl, hi = below + incl;
    const unsigned own = __ballot_sync(0xffffffffu, t > lo && t <= hi);
    const int src = own ? __ffs(own) - 1 : 0;
    *base = __shfl_sync(0xffffffffu, lo, src);
    return own ? src : -1;
}
// The same for a re-draw, where the token must exist: the first lane with mass whose running sum reaches the target,
// or by rounding the last lane with mass (-1: no lane has any).
__device__ __forceinline__ int pick_lane(double v, double below, double t, double* base, double* total, bool* hit) {
    const int lane = threadIdx.x & 31;
    double incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) { const double t2 = shfl_up_d(incl, o); if (lane >= o) incl += t2; }
    double excl = shfl_up_d(incl, 1);
    if (lane == 0) excl = 0.0;
    *total = below + __shfl_sync(0xffffffffu, incl, 31);
    const unsigned has = __ballot_sync(0xffffffffu, v > 0.0), reach = __ballot_sync(0xffffffffu, v > 0.0 && below + incl >= t);
    *hit = reach != 0;
    const int src = reach ? __ffs(reach) - 1 : (has ? 31 - __clz(has) : 0);
    *base = below + __shfl_sync(0xffffffffu, excl, src);
    return has ? src : -1;
}

__device__ const double g_pow2_64[64] = {      // 2^(j/64)
    1.0, 1.0108892860517005, 1.0218971486541166, 1.0330248790212284,
    1.0442737824274138, 1.0556451783605572, 1.0671404006768237, 1.0787607977571199,
    1.0905077326652577, 1.102382583307841, 1.1143867425958924, 1.1265216186082418,
    1.1387886347566916, 1.1511892299529827, 1.1637248587775775, 1.1763969916502812,
    1.189207115002721, 1.202156731452703, 1.215247359980469, 1.22848053610687,
    1.241857812073484, 1.255380757024691, 1.2690509571917332, 1.2828700160787783,
    1.2968395546510096, 1.3109612115247644, 1.3252366431597413, 1.339667524053303,
    1.3542555469368927, 1.3690024229745905, 1.383909881963832, 1.3989796725383112,
    1.4142135623730951, 1.42961333839197, 1.4451808069770467, 1.460917794180647,
    1.4768261459394993, 1.4929077282912648, 1.5091644275934228, 1.5255981507445384,
    1.5422108254079407, 1.559004400237837, 1.5759808451078865, 1.593142151342267,
    1.6104903319492543, 1.6280274218573478, 1.645755478153965, 1.6636765803267364,
    1.681792830507429, 1.7001063537185235, 1.718619298122478, 1.7373338352737062,
    1.7562521603732995, 1.7753764925265212, 1.7947090750031072, 1.8142521755003989,
    1.8340080864093424, 1.8539791250833855, 1.8741676341103, 1.8945759815869656,
    1.9152065613971474, 1.9360617934922943, 1.9571441241754002, 1.978456026387951,
};
// 2^t in double for t <= about 0: t = n/64 + f with |f| <= 1/128, 2^t = 2^(n >> 6) * tab[n & 63] * 2^f, 2^f by its
// series to the fifth power (the next term is below 4e-17 of the result).  `tab` holds 2^(j/64), j = 0..63.  Arguments
// below -1000 (and -inf) give 0.
__device__ __forceinline__ double q_exp2(double t, const double* tab) {
    const double magic = 6755399441055744.0;                 // 1.5 * 2^52: adding it rounds to an integer
    const double tm = fma(t, 64.0, magic);
    const int n = __double2loint(tm);
    const double f = fma(tm - magic, -1.0 / 64.0, t);         // exact
    double p = fma(f, 0.0013333558146428443, 0.009618129107628477);     // ln2^5/120, ln2^4/24
    p = fma(f, p, 0.05550410866482158);                                 // ln2^3/6
    p = fma(f, p, 0.2402265069591007);                                  // ln2^2/2
    p = fma(f, p, 0.6931471805599453);                                  // ln2
    const double s = tab[n & 63];
    const double r = fma(s * f, p, s);
    const int keep = t > -1000.0 ? -1 : 0;                   // (a mask: as a choice of doubles it became a branch around all of the above)
    return __hiloint2double((__double2hiint(r) + ((n >> 6) << 20)) & keep, __double2loint(r) & keep);
}

}  // namespace

}  // namespace bebop
