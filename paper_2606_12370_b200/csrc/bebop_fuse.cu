// Fused kernel: bebop_tv and bebop_verify (with its TV output) as the stream of bebop_flow.cuh.
#include "bebop_flow.cuh"
#include <type_traits>

namespace bebop {

template <int DT, bool TVM, class F>
__global__ void __launch_bounds__(F::LT, 1) k_fuse(const __grid_constant__ FlowArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    flow_body<DT, TVM, F>(a, smem);
}

cudaError_t fuse_verify(const RowArgs& a, const Plan& p, const int32_t* draft_tokens, const float* u_accept,
                        const float* u_final, VerifyOut o, char* ws, cudaStream_t stream, bool* launched, bool tv_only,
                        float* s_aux, bool large_chunks) {
    const FlowCall x{a, p, draft_tokens, u_accept, u_final, o, ws, stream, tv_only, s_aux};
    const int C = flow_cluster(a, tv_only);
    const bool big = large_chunks || flow_long(a, tv_only, C);
    const auto go = [&](auto dt, auto tvm) {
        // (bebop_tv of such rows is the sequence kernel's)
        if constexpr (!tvm.value) if (!large_chunks && flow_resident_rows(a, C)) return flow_launch<FlowResident, k_fuse<dt.value, tvm.value, FlowResident>>(x, C, launched);
        return big ? flow_launch<FlowLong, k_fuse<dt.value, tvm.value, FlowLong>>(x, C, launched)
                   : flow_launch<FlowShort, k_fuse<dt.value, tvm.value, FlowShort>>(x, C, launched);
    };
    using F32 = std::integral_constant<int, 0>;
    using BF16 = std::integral_constant<int, 1>;
    if (tv_only) return a.dt == 0 ? go(F32{}, std::true_type{}) : go(BF16{}, std::true_type{});
    return a.dt == 0 ? go(F32{}, std::false_type{}) : go(BF16{}, std::false_type{});
}

// With TV both names run the stream, by the same rules for clusters and chunks, and the line only says under which name a call
// goes: bebop_tv up to 32 slices of 1024 vectors per row, bebop_verify up to eight slices (fp32: six), with one draft position, or up to 40
// (row, slice) tasks per SM.  Without TV (us per call on a B200, bf16) the sweeps read one row
// per sequence twice and the stream all of them: calls of up to 40 tasks per SM go through the stream (64 of 151,936 logits 73
// against 77, 24 47 against 53), rows of two or three slices with up to four positions (1,000 of 16,000, K = 2, 89 against 108; 400 of
// 24,000, K = 4, 79 against 85), and rows that stay resident (1,000 of 8,000, K = 8, 131 against 140, 1,000 of 5,000 fp32, K = 8, 107 against 137,
// 1,000 of 12,288, K = 8, 143 against 142); the others through the sweeps (192 of 32,000, K = 7, 74 against 95; 300 of 65,536 97 against
// 106).
bool fuse_preferred(const RowArgs& a, bool tv_only, bool want_tv) {
    const int T = (a.nvec + 1023) / 1024;
    int sms = 0, dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) { cudaGetLastError(); return false; }
    const long long tasks = (long long)a.B * (tv_only ? 1 : a.K + 1) * T;
    if (T > 32 || tasks < 2LL * sms) return false;
    if (tv_only) return true;
    if (want_tv && (T <= (a.dt == 0 ? 6 : 8) || a.K == 1)) return true;
    return tasks <= 40LL * sms || (!want_tv && ((a.K <= 4 && (T == 2 || T == 3)) || flow_resident_rows(a, flow_cluster(a, false))));
}

}  // namespace bebop
