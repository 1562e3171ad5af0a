// Fused evaluation pass: k-of-W exceedance counts, robust deviation score, per-metric
// threshold and persistence, the multi-signal flag with the step-time metric as primary
// signal, the response tier and the consecutive-evaluation counter.
#include "kernels.h"

namespace guard {

namespace {

// A CTA scores the ranks whose exceedance entries are LW words of 32 bits of a ring row: 128 or 32 ranks of byte-wide
// entries (at most 8 metrics), 32 or 8 ranks of word-wide ones.  Its warps split the window's steps, 32 / LW steps per
// warp and load; acc[i] += (word >> i) & 0x01010101 counts bits i, i + 8, i + 16 and i + 24 of a lane's word in its byte
// lanes: metric i of four ranks, or metrics i, i + 8, ... of one.  The warps' counts meet in shared memory, in halves of
// 16 bits.  Then a thread per (rank, metric), coalesced, and one per rank.
// The counts need only the exceedance rows, so they are taken before the wait for the fleet baseline in front: this
// kernel starts beside it.  Bound by the latency of the row loads (eight in flight per lane), which that hides, then by
// the chain baseline - score - store: at 16 384 ranks x 8 metrics x 200 steps it ends 3.2 us after the baseline, at
// 4 096 x 16 x 120 2.5 us (10.5 and 40 us with a launch behind the baseline, a thread per rank and, for words, one load
// in flight).
template <int MB, int NM, int LW>      // bytes per entry; metrics if known (a power of two), else 0; words of a row
__global__ void __launch_bounds__(1024, 1) score_flag_kernel(const ScoreArgs a, const MetricParams p) {
    constexpr int kRanks = LW * 4 / MB, RW = 32 / LW;
    __shared__ float s_B[kMaxMetrics], s_rhs[kMaxMetrics], s_Ds[kMaxMetrics];
    __shared__ uint32_t s_cnt[8][2][LW], s_left[8][2][LW];   // bits i + 16 j: [i][0], i + 8 + 16 j: [i][1], j the halves
    __shared__ uint32_t s_mask[kRanks];
    __shared__ float s_dev[kRanks];
    const int M = NM ? NM : a.M, tid = threadIdx.x, T = blockDim.x, lane = lane_id(), row = tid / LW, rows = T / LW;   // this thread's first step, steps per round
    if (a.topk_idx && blockIdx.x == gridDim.x - 1) {         // the ranks a top-k selection has picked, and their scores
        pdl_wait();
        const int pm = p.primary;
        const float B = a.fleet_med[pm], Ds = scale_of(a.fleet_mad[pm], B, p.floor_rel[pm], p.floor_abs[pm]);
        for (int i = tid; i < a.K; i += T) {
            const int32_t r = a.topk_idx[i];
            float dev = __fsub_rn(a.wmed[(size_t)r * M + pm], B);
            if (p.dir[pm] < 0) dev = -dev;
            if (a.topk_user) a.topk_user[i] = r;
            if (a.topk_score) a.topk_score[i] = (dev == 0.0f) ? 0.0f : __fdiv_rn(__fmul_rn(0.6745f, dev), Ds);
        }
        pdl_trigger();
        return;
    }
    const int r0 = blockIdx.x * kRanks, nr = min(kRanks, a.R - r0);
    for (int i = tid; i < 16 * LW; i += T) { (&s_cnt[0][0][0])[i] = 0u; (&s_left[0][0][0])[i] = 0u; }
    for (int i = tid; i < kRanks; i += T) s_mask[i] = 0u;
    __syncthreads();

    const char *base = (const char *)a.mask_base + (size_t)r0 * MB;
    const size_t pitch = (size_t)a.R * MB;
    const int first = a.last_slot - (a.n - 1) + (a.last_slot < a.n - 1 ? a.capacity : 0);
    const int at = 4 * (lane % LW), bytes = nr * MB;                // this lane's bytes of a row's share
    const bool word_ok = at + 4 <= bytes && (pitch & 3) == 0;
    auto load = [&](int slot) -> uint32_t {
        const char *q = base + (size_t)slot * pitch + at;
        if (word_ok) return __ldg(reinterpret_cast<const uint32_t *>(q));
        uint32_t v = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b)
            if (at + b < bytes) v |= (uint32_t)(uint8_t)q[b] << (8 * b);
        return v;
    };
    uint32_t acc[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = 0u;
    auto merge = [&](uint32_t (&to)[8][2][LW]) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            uint32_t even = acc[i] & 0x00FF00FFu, odd = (acc[i] >> 8) & 0x00FF00FFu;
#pragma unroll
            for (int d = LW; d < 32; d <<= 1) {
                even += __shfl_xor_sync(0xFFFFFFFFu, even, d);
                odd += __shfl_xor_sync(0xFFFFFFFFu, odd, d);
            }
            if (even && lane < LW) atomicAdd(&to[i][0][lane], even);
            if (odd && lane < LW) atomicAdd(&to[i][1][lane], odd);
            acc[i] = 0u;
        }
    };
    if (a.slide) {
        // the steps that entered, then those that left (up to eight each)
        auto pass = [&](const int from, const int steps, uint32_t (&to)[8][2][LW]) {
            for (int j0 = (row / RW) * RW; j0 < steps; j0 += rows) {     // (the same for a whole warp)
                const int j = j0 + row % RW;
                int slot = from + j;
                if (slot < 0) slot += a.capacity;
                const uint32_t word = j < steps ? load(slot) : 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] = (word >> i) & 0x01010101u;
                merge(to);
            }
        };
        pass(a.last_slot - (a.entering - 1), a.entering, s_cnt);
        pass(first - a.leaving, a.leaving, s_left);
    } else {
        constexpr int KU = 8;  // loads in flight per lane
        int held = 0;
        for (int j0 = (row / RW) * RW; j0 < a.n; j0 += rows * KU) {      // (the same for a whole warp)
            uint32_t word[KU];
#pragma unroll
            for (int u = 0; u < KU; ++u) {
                const int j = j0 + row % RW + u * rows;
                int slot = first + j;
                if (slot >= a.capacity) slot -= a.capacity;
                word[u] = j < a.n ? load(slot) : 0u;
            }
#pragma unroll
            for (int u = 0; u < KU; ++u)
#pragma unroll
                for (int i = 0; i < 8; ++i) acc[i] += (word[u] >> i) & 0x01010101u;
            held += KU;
            if (held > 255 - KU) { merge(s_cnt); held = 0; }   // a byte is about to overflow
        }
        merge(s_cnt);
    }
    // (the medians are complete before the baseline in front starts, which reads them, and so is the caller's earlier work on
    // its copy: written here, where it hides behind the baseline; a block of 32 steps of 136 ranks x 8 and its evaluation
    // take 27.0 us when it is written beside the scores, 26.2 so)
    if (a.wmed_user)
        for (int e = tid; e < nr * M; e += T) a.wmed_user[(size_t)r0 * M + e] = a.wmed[(size_t)r0 * M + e];
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    if (tid < M) {
        const float B = a.fleet_med[tid], Ds = scale_of(a.fleet_mad[tid], B, p.floor_rel[tid], p.floor_abs[tid]);
        s_B[tid] = B;
        s_Ds[tid] = Ds;
        s_rhs[tid] = __fmul_rn(p.thrp[tid], Ds);
    }
    __syncthreads();
    for (int e = tid; e < nr * M; e += T) {
        const int rl = e / M, m = e - rl * M;
        const size_t o = (size_t)r0 * M + e;
        const float x = a.wmed[o];
        // byte lane q of acc[i]: rank 4 lane + q, metric i / rank `lane`, metric i + 8 q
        const int i = MB == 1 ? m : m & 7, q = MB == 1 ? rl & 3 : m >> 3, l = MB == 1 ? rl >> 2 : rl;
        int cnt = (int)((s_cnt[i][q & 1][l] >> (16 * (q >> 1))) & 0xFFFFu);
        if (a.slide) cnt += (int)a.kcnt[o] - (int)((s_left[i][q & 1][l] >> (16 * (q >> 1))) & 0xFFFFu);
        if (a.kcnt) a.kcnt[o] = (uint16_t)cnt;
        float dev = __fsub_rn(x, s_B[m]);
        if (p.dir[m] < 0) dev = -dev;
        if (dev > s_rhs[m] && cnt >= p.k) atomicOr(&s_mask[rl], 1u << m);
        if (m == p.primary) s_dev[rl] = dev;
        if (a.counts) a.counts[o] = (uint16_t)cnt;
        if (a.scores) a.scores[o] = (dev == 0.0f) ? 0.0f : __fdiv_rn(__fmul_rn(0.6745f, dev), s_Ds[m]);
    }
    __syncthreads();
    const int need = min(p.min_signals, M);
    for (int rl = tid; rl < nr; rl += T) {
        const int r = r0 + rl;
        const uint32_t mask = s_mask[rl];
        const bool cand = ((mask >> p.primary) & 1u) && (__popc(mask) >= need);
        int c = a.consec[r];
        c = cand ? min(c + 1, 255) : 0;
        a.consec[r] = (uint8_t)c;
        const bool flag = cand && (c >= p.n_consec);
        const float absB = fabsf(s_B[p.primary]);
        int t = 0;
        if (flag && s_dev[rl] >= __fmul_rn(p.tier_severe, absB)) t = 3;
        else if (flag && s_dev[rl] >= __fmul_rn(p.tier_moderate, absB)) t = 2;
        else if (mask != 0) t = 1;
        if (a.metric_mask) a.metric_mask[r] = mask;
        if (a.flags) a.flags[r] = (uint8_t)flag;
        if (a.tier) a.tier[r] = (uint8_t)t;
        a.flags_keep[r] = (uint8_t)flag;
        a.tier_keep[r] = (uint8_t)t;
    }
}

// Node-level fold.  A CTA takes 32 nodes; its eight warps split the window's steps (warp w takes
// steps w, w + 8, ...), lane l owns node l of the CTA's 32.  "All ranks of the node exceeded on the
// primary metric in this step" is an AND over the node's exceedance entries; with eight ranks per
// node and byte-wide entries that is one 64-bit load and one mask test.
constexpr int kNodeWarps = 8;

template <typename MaskT>
__global__ void __launch_bounds__(kNodeWarps * 32) node_verdict_kernel(const NodeArgs a) {
    __shared__ uint32_t s_stall[32];
    const int lane = lane_id(), w = warp_id();
    const int node = blockIdx.x * 32 + lane;
    if (threadIdx.x < 32) s_stall[threadIdx.x] = 0;
    __syncthreads();
    const bool live = node < a.nodes;
    const int rpn = a.ranks_per_node;
    const size_t r0 = (size_t)node * rpn;
    const MaskT *mask_base = (const MaskT *)a.mask_base;
    const int first = a.last_slot - (a.n - 1) + (a.last_slot < a.n - 1 ? a.capacity : 0);
    const bool wide = sizeof(MaskT) == 1 && rpn == 8 && (a.R & 7) == 0;
    const unsigned long long want = 0x0101010101010101ull << a.primary;
    uint32_t stall = 0;
    if (live) {
        for (int j = w; j < a.n; j += kNodeWarps) {
            int slot = first + j;
            if (slot >= a.capacity) slot -= a.capacity;
            const MaskT *rowp = mask_base + (size_t)slot * a.R + r0;
            bool all = true;
            if (wide) {
                all = (__ldg(reinterpret_cast<const unsigned long long *>(rowp)) & want) == want;
            } else {
                for (int q = 0; q < rpn; ++q) all = all && (((uint32_t)rowp[q] >> a.primary) & 1u);
            }
            stall += all;
        }
        if (stall) atomicAdd(&s_stall[lane], stall);
    }
    __syncthreads();
    pdl_wait();                    // (the stall counts need only the exceedance rows; flags and tiers come from the score pass in front)
    if (w == 0 && live) {
        int any = 0, top = 0;
        for (int q = 0; q < rpn; ++q) {
            any |= a.flags[r0 + q];
            top = max(top, (int)a.tier[r0 + q]);
        }
        if (a.node_flag) a.node_flag[node] = (uint8_t)(any != 0);
        if (a.node_tier) a.node_tier[node] = (uint8_t)top;
        if (a.node_stall) a.node_stall[node] = (uint16_t)s_stall[lane];
    }
}

}  // namespace

cudaError_t launch_node_verdict(const NodeArgs &a, cudaStream_t st) {
    const int grid = (a.nodes + 31) / 32;
    if (a.mask_bytes == 1) return launch_after(node_verdict_kernel<uint8_t>, grid, kNodeWarps * 32, st, a);
    return launch_after(node_verdict_kernel<uint32_t>, grid, kNodeWarps * 32, st, a);
}

template <int LW>
static cudaError_t launch_score(const ScoreArgs &a, const MetricParams &p, cudaStream_t st) {
    const int ranks = LW * 4 / a.mask_bytes, grid = (a.R + ranks - 1) / ranks + (a.topk_idx ? 1 : 0);
    // threads: eight loads each while one CTA can have them; where the CTAs fill the GPU anyway, 32 (larger ones keep SMs
    // from the kernels of the next evaluation: passes of 200 x 16 384 x 8 with overlapped evaluations take 433 us with
    // 256 threads per CTA, 436 with 512, 447 with 1 024)
    int T = 256;
    while (T < 1024 && !a.slide && (long long)a.n * LW > (LW == 32 ? 32LL : 8LL) * T) T <<= 1;
    if (a.mask_bytes != 1) return launch_after(score_flag_kernel<4, 0, LW>, grid, T, st, a, p);
    if (a.M == 8) return launch_after(score_flag_kernel<1, 8, LW>, grid, T, st, a, p);
    return launch_after(score_flag_kernel<1, 0, LW>, grid, T, st, a, p);
}

cudaError_t launch_score_flag(const ScoreArgs &a, const MetricParams &p, cudaStream_t st) {
    // full cache lines of a row where that makes a CTA for every other SM, else sectors of it and four times the CTAs
    // (1 024 ranks, 1 000 steps: 7.1 us beside and behind the baseline against 12.8; 8 192 ranks, 100 steps: the same)
    return (long long)a.R * a.mask_bytes > 74 * 128 ? launch_score<32>(a, p, st) : launch_score<8>(a, p, st);
}

}  // namespace guard
