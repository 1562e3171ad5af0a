// Cross-rank selection of whole rows held in registers (xrank_count.cuh): the path of small and middle fleets,
// of other numbers of metrics than the streaming sweeps take, and of single rows.
#include "xrank_count.cuh"

namespace guard {

namespace {

template <int V, int C>
__global__ void __launch_bounds__(1024) xrank_count_kernel(const XrankArgs a, const MetricParams p) {
    __shared__ CtShared<C> sh;
    pdl_wait();
    ct_row<V, C>(a, p, blockIdx.y, blockIdx.x * C, sh);
}

// A cluster of NC CTAs per column: a few wide columns.
template <int V, int NC, bool APART>
__global__ void __cluster_dims__(NC, 1, 1) __launch_bounds__(ct_most_threads(NC), 512 / ct_most_threads(NC)) xrank_count_cluster_kernel(const XrankArgs a, const MetricParams p) {
    __shared__ CtShared<1> sh;
    pdl_wait();
    const int column = (int)blockIdx.x / NC;
    if (APART) ct_row<V, 1, NC>(a, p, blockIdx.y, column % a.M, sh, column < a.M ? kCtStatistics : kCtCut);
    else ct_row<V, 1, NC>(a, p, blockIdx.y, column, sh);
    ct_sync<NC>();   // the other CTAs read this one's lists last: none may exit before all have
}

// One row's median and MAD, and beside them its extra order statistic, a CTA each (R <= 4 blockDim.x).
__global__ void __launch_bounds__(1024) xrank_count_apart_kernel(const XrankArgs a, const MetricParams p) {
    __shared__ CtShared<1> sh;
    pdl_wait();
    ct_row<4, 1>(a, p, 0, (int)blockIdx.x % a.M, sh, (int)blockIdx.x < a.M ? kCtStatistics : kCtCut);
}

template <int NC, bool APART>
cudaError_t launch_cluster(const XrankArgs &a, const MetricParams &p, int S, cudaStream_t st) {
    const dim3 grid(a.M * NC * (APART ? 2 : 1), S);
    const int T = ct_cluster_threads(a.R, NC, ct_most_threads(NC));
    const int v = (a.R + NC * T - 1) / (NC * T);
    if (v <= 4) return launch_after(xrank_count_cluster_kernel<4, NC, APART>, grid, T, st, a, p);
    if (v <= 8) return launch_after(xrank_count_cluster_kernel<8, NC, APART>, grid, T, st, a, p);
    return launch_after(xrank_count_cluster_kernel<16, NC, APART>, grid, T, st, a, p);
}

template <int C>
cudaError_t launch_c(const XrankArgs &a, const MetricParams &p, int S, int T, cudaStream_t st) {
    const int v = (a.R * C + T - 1) / T;
    const dim3 grid(a.M / C, S);
    if (v <= 4) return launch_after(xrank_count_kernel<4, C>, grid, T, st, a, p);
    if (v <= 8) return launch_after(xrank_count_kernel<8, C>, grid, T, st, a, p);
    if (v <= 16) return launch_after(xrank_count_kernel<16, C>, grid, T, st, a, p);
    return launch_after(xrank_count_kernel<32, C>, grid, T, st, a, p);
}

constexpr int kGridRows = 65535;   // the largest grid in y: rows per launch

// Metrics and threads per CTA.
void plan(const int R, const int M, const int S, int &C, int &T) {
    // Two metrics per CTA where that leaves at least a CTA per SM (their loads share cache lines; more metrics make
    // larger CTAs, which wait longer at their barriers: 60 steps of 4 096 ranks x 16 metrics take 31 / 29 / 29 us, launch
    // included, with 1 / 2 / 8 of them, 100 steps of 1 024 x 8 take 14 / 14 / 18), else one.
    C = (M % 2 == 0 && 2 * R <= kCountMaxRanks && (long long)S * (M / 2) >= 148) ? 2 : 1;
    const long long ctas = (long long)S * (M / C);
    const int E = R * C;
    // threads: few values each while the CTAs are few (a pass is then as short as it gets), else CTAs small enough to
    // share an SM and hide one another's barriers
    T = 32 * C;
    if (ctas <= 148) { while (T < 1024 && E > 4 * T) T <<= 1; }
    else { while (T < 256 && E > 8 * T) T <<= 1; }
    while (T < 1024 && E > 32 * T) T <<= 1;
}

}  // namespace

int xrank_count_launches(int S) { return (S + kGridRows - 1) / kGridRows; }

bool xrank_count_supported(int R) { return R >= 1 && R <= kCountMaxRanks; }

bool xrank_count_copies(int R, int M, int S) {
    if (R > kCtClusterRanks) return false;
    int C, T;
    plan(R, M, S, C, T);
    return (long long)R * C <= 8LL * T;
}

cudaError_t launch_xrank_count(const XrankArgs &a, const MetricParams &p, int S, cudaStream_t st) {
    if (S <= 0) return cudaSuccess;
    // few and wide columns: a cluster each, of the most CTAs that find an SM each
    // An extra order statistic by CTAs of its own, beside median and MAD, where they find SMs too (a sweep's fleet
    // statistics, 6 metrics of 16 384 GPUs: 13.2 us, one after the other 18.5; 296 GPUs 5.9 and 8.6).
    const long long columns = (long long)S * a.M;
    if (a.R > kCtClusterRanks && columns * 4 <= 148) {
        if (a.cut && columns * 16 <= 148) return launch_cluster<8, true>(a, p, S, st);
        if (a.cut && columns * 8 <= 148) return launch_cluster<4, true>(a, p, S, st);
        return columns * 8 <= 148 ? launch_cluster<8, false>(a, p, S, st) : launch_cluster<4, false>(a, p, S, st);
    }
    int C, T;
    plan(a.R, a.M, S, C, T);
    if (a.cut && S == 1 && C == 1 && a.R <= 4 * T) return launch_after(xrank_count_apart_kernel, 2 * a.M, T, st, a, p);
    XrankArgs g = a;
    for (int s0 = 0; s0 < S; s0 += kGridRows) {
        const int n = S - s0 < kGridRows ? S - s0 : kGridRows;
        const size_t o = (size_t)s0 * a.M;
        g.first_slot = (int)(((long long)a.first_slot + s0) % a.capacity);
        g.copy_from = a.copy_from ? a.copy_from + (size_t)s0 * a.row_stride : nullptr;
        g.med = a.med + o;
        g.mad = a.mad + o;
        g.med_user = a.med_user ? a.med_user + o : nullptr;
        g.mad_user = a.mad_user ? a.mad_user + o : nullptr;
        g.prev_rows = a.prev_rows > s0 ? a.prev_rows - s0 : 0;
        const cudaError_t e = C == 2 ? launch_c<2>(g, p, n, T, st) : launch_c<1>(g, p, n, T, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace guard
