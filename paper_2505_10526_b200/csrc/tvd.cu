// Total variation distance between the target's and the drafter's token
// distributions for every drafted position (paper Eq. 6):
//     TVD(p_j, q_j) = 1/2 * sum_v |p_j(v) - q_j(v)|,      p_j = softmax(z_j / T)
// and the acceptance probability of the rejection test, sum_v min(p_j(v), q_j(v)) = 1 - TVD.
// Every reduction has a fixed order.
//   tvd_row_kernel     a row in the shared memory of a cluster of CTAs: the logits cross HBM once whether or not the
//                      caller hands in the statistics the acceptance call left behind.
// For more rows than are resident that way, three kernels:
//   tvd_stream_kernel  twice: max logit and sum of exponentials of every row (skipped when the statistics are given), then
//                      the sums of |p-q| and min(p,q);
//   tvd_final_kernel   adds a row's shares in order.
#include "kernels.cuh"
#include "ptx.cuh"

namespace massv {

namespace {

// Row r of the drafted positions = (sequence b, draft j): logits row b*(gamma+1)+j, q row b*gamma+j.
__device__ __forceinline__ const float* logits_row(const TvdParams& p, int row) {
    const int b = row / p.gamma, j = row % p.gamma;
    return p.logits + (size_t)(b * (p.gamma + 1) + j) * p.V;
}

__device__ __forceinline__ void bulk_load_1d_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t policy) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
                 : "memory");
}

// Two persistent passes, one CTA per SM: statistics (max and sum of exponentials of the logits), then the sums of |p - q|
// and min(p, q).  What bounds them: HBM (4 and 8 B per entry), and close behind it the issue of about 17 instructions per
// entry, so nothing is computed per step that can wait.  The rows' steps of 6,144 entries form one line; every CTA takes
// an equal contiguous run of it, meets two or three rows and reduces over its threads only where a row ends.  A producer
// warp keeps a ring of steps filled with bulk copies (two groups of four entries per consumer thread and step), so the
// bytes in flight do not depend on what the consumers do.  The second pass walks the rows last to first: the statistics
// pass has left the last logits in L2, and the drafter's rows pass through without displacing them.  64 x 5 rows of
// 152,064, calls back to back: 136 us with a grid of (slice, row) CTAs and one 16-byte load per thread and iteration, 112 us
// here (44 - 49 us of it the first pass).
constexpr int kStreamWarps = 24;                             // consumers
constexpr int kStreamConsumers = kStreamWarps * 32, kStreamThreads = kStreamConsumers + 32;
constexpr int kStepGroups = 2;
constexpr int kStepEntries = kStepGroups * 4 * kStreamConsumers;
constexpr int kStreamStages = 4;                             // of the second pass (logits and q); the first has twice as many
constexpr int kStreamSmem = kStreamStages * 2 * kStepEntries * 4;

// The pieces of a row: CTA c of the line takes steps [c * per, (c + 1) * per).  A row's result of either pass is up to
// kTvdSlices shares, one per CTA that met it.
struct RowShares {
    int first_cta, n;
    __device__ RowShares(int line_row, int steps_per_row, int per) {
        first_cta = line_row * steps_per_row / per;
        n = ((line_row + 1) * steps_per_row - 1) / per - first_cta + 1;
    }
};
// A position on the line, moved step by step.
struct StreamPos {
    int row, step;                        // row along the line; step inside the row
    __device__ StreamPos(int at, int steps_per_row) : row(at / steps_per_row), step(at % steps_per_row) {}
    __device__ __forceinline__ void advance(int steps_per_row) { if (++step == steps_per_row) { step = 0; ++row; } }
};
__device__ __forceinline__ void consumers_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kStreamConsumers) : "memory"); }

// SUM = false: the statistics pass, ring of 2 * kStreamStages steps of logits.  SUM = true: the second pass, ring of
// kStreamStages steps of logits and q.
template <bool SUM>
__global__ void __launch_bounds__(kStreamThreads, 1) tvd_stream_kernel(TvdParams p, int steps_per_row, int per) {
    constexpr int kStages = SUM ? kStreamStages : 2 * kStreamStages;
    constexpr int kStageEntries = SUM ? 2 * kStepEntries : kStepEntries;
    extern __shared__ __align__(128) float ring[];              // [kStages][logits(, q)]
    __shared__ __align__(8) uint64_t full_bar[kStages], empty_bar[kStages];
    __shared__ double s_a[kStreamWarps], s_b[kStreamWarps];
    __shared__ float s_m[kStreamWarps];
    __shared__ int s_abort;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rows = p.B * p.gamma, at0 = (int)blockIdx.x * per, n_steps = min(per, rows * steps_per_row - at0);      // >= 1
    if (t == 0) {
        for (int s = 0; s < kStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], kStreamWarps); }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // Behind the statistics pass the inputs are complete (its CTAs let this grid start only after their own wait): the
    // second pass's copies need not wait for its results.  Behind the acceptance call they are that call's outputs.
    const bool wait_first = !SUM || p.row_stats != nullptr;
    if (wait_first) pdl_wait();
    volatile int* abort_ptr = &s_abort;
    StreamPos pos(at0, steps_per_row);

    if (warp == kStreamWarps) {
        // ------------------------------------------------ producer
        if (wait_first) pdl_trigger();
        if (lane == 0) {
            uint64_t pass;
            asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pass));
            int stage = 0;
            uint32_t ph = 0;
            bool ok = true;
            for (int s = 0; s < n_steps && ok; ++s) {
                if (!mbar_wait(&empty_bar[stage], ph ^ 1u, abort_ptr)) { ok = false; break; }
                const int row = SUM ? rows - 1 - pos.row : pos.row, e0 = pos.step * kStepEntries;
                const uint32_t bytes = (uint32_t)min(kStepEntries, p.V - e0) * 4u;       // V is a multiple of 8
                float* dst = ring + stage * kStageEntries;
                mbar_expect_tx(&full_bar[stage], SUM ? 2 * bytes : bytes);
                bulk_load_1d(dst, logits_row(p, row) + e0, bytes, &full_bar[stage]);
                if (SUM) bulk_load_1d_hint(dst + kStepEntries, p.draft_probs + (size_t)row * p.V + e0, bytes, &full_bar[stage], pass);
                pos.advance(steps_per_row);
                if (++stage == kStages) { stage = 0; ph ^= 1u; }
            }
            if (!ok) {
                for (int i = 0; i < 64; ++i) __nanosleep(2000);       // let copies in flight land
                set_status(p.dev_status, MASSV_ERR_TIMEOUT);
            }
        }
        if (!wait_first) { pdl_wait(); pdl_trigger(); }
        return;
    }
    // ---------------------------------------------------- consumers (a wait that gave up leaves the abort flag and
    // goes on: every warp meets the same barriers)
    if (!wait_first) pdl_wait();
    pdl_trigger();
    int stage = 0;
    uint32_t ph = 0;
    float4 x[kStepGroups], y[kStepGroups];
    // the step's groups of this thread into registers (nothing past the row's end), and the stage back to the producer
    auto take = [&](int step) {
        if (!mbar_wait_warp(&full_bar[stage], ph, abort_ptr) && lane == 0) set_status(p.dev_status, MASSV_ERR_TIMEOUT);
        const float4* src = reinterpret_cast<const float4*>(ring + stage * kStageEntries);
        const int left = p.V / 4 - step * (kStepEntries / 4);
#pragma unroll
        for (int k = 0; k < kStepGroups; ++k) {
            const int i = t + k * kStreamConsumers;
            x[k] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            if (SUM) y[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (i < left) {
                x[k] = src[i];
                if (SUM) y[k] = src[kStepEntries / 4 + i];
            }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty_bar[stage]);
        if (++stage == kStages) { stage = 0; ph ^= 1u; }
    };
    if constexpr (!SUM) {
        float m = -INFINITY;              // this thread's running maximum and its sum relative to it
        double sum = 0.0;
        for (int s = 0; s < n_steps; ++s) {
            take(pos.step);
            float top = m;
#pragma unroll
            for (int k = 0; k < kStepGroups; ++k) top = fmaxf(top, fmaxf(fmaxf(x[k].x, x[k].y), fmaxf(x[k].z, x[k].w)));
            if (top > m) {                // (rare after a row's first steps)
                if (m > -INFINITY) sum *= (double)expf((m - top) * p.inv_T);
                m = top;
            }
            const float ref = m == -INFINITY ? 0.f : m;      // nothing finite so far: weights of zero
#pragma unroll
            for (int k = 0; k < kStepGroups; ++k)
                sum += (double)((expf((x[k].x - ref) * p.inv_T) + expf((x[k].y - ref) * p.inv_T)) +
                                (expf((x[k].z - ref) * p.inv_T) + expf((x[k].w - ref) * p.inv_T)));
            const int row = pos.row;
            pos.advance(steps_per_row);
            if (s + 1 < n_steps && pos.row == row) continue;
            // the end of the row, or of this CTA's run
            float wm = m;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) wm = fmaxf(wm, __shfl_xor_sync(0xffffffffu, wm, o));
            double ws = m == -INFINITY ? sum : sum * (double)expf((m - wm) * p.inv_T);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) ws += __shfl_xor_sync(0xffffffffu, ws, o);
            if (lane == 0) { s_m[warp] = wm; s_a[warp] = ws; }
            consumers_sync();
            if (warp == 0) {
                const float lm = lane < kStreamWarps ? s_m[lane] : -INFINITY;
                float M = lm;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                double S = lane < kStreamWarps ? s_a[lane] : 0.0;
                if (lm != -INFINITY) S *= (double)expf((lm - M) * p.inv_T);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
                const int share = (int)blockIdx.x - RowShares(row, steps_per_row, per).first_cta;
                if (lane == 0) {
                    p.slice_max[row * kTvdSlices + share] = M;
                    p.slice_sum[row * kTvdSlices + share] = S;
                }
            }
            consumers_sync();
            m = -INFINITY; sum = 0.0;
        }
    } else {
        double a = 0.0, mn = 0.0;
        float M = 0.f, inv_sum = 0.f;
        int cur = -1;                     // the row (along the line) whose statistics are in M, inv_sum
        for (int s = 0; s < n_steps; ++s) {
            const int row = rows - 1 - pos.row;
            if (cur != pos.row) {
                cur = pos.row;
                double S;
                if (p.row_stats) {
                    // the acceptance scan's merged statistics of logits row b*(gamma+1)+j
                    const int b = row / p.gamma, j = row % p.gamma;
                    const float2 ms = *reinterpret_cast<const float2*>(p.row_stats + (size_t)(b * (p.gamma + 1) + j) * 2);
                    M = ms.x;
                    S = (double)ms.y;
                } else {
                    const int n = RowShares(row, steps_per_row, per).n;          // (the statistics pass walked the rows in order)
                    const float ms = lane < n ? p.slice_max[row * kTvdSlices + lane] : -INFINITY;
                    M = ms;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
                    S = lane < n ? p.slice_sum[row * kTvdSlices + lane] : 0.0;
                    if (ms != -INFINITY) S *= (double)expf((ms - M) * p.inv_T);
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
                }
                inv_sum = (float)(1.0 / S);
            }
            take(pos.step);
#pragma unroll
            for (int k = 0; k < kStepGroups; ++k) {
                const float e[4] = {x[k].x, x[k].y, x[k].z, x[k].w}, f[4] = {y[k].x, y[k].y, y[k].z, y[k].w};
                float fa = 0.f, fm = 0.f;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float pv = expf((e[j] - M) * p.inv_T) * inv_sum;
                    fa += fabsf(pv - f[j]);
                    fm += fminf(pv, f[j]);
                }
                if (t + k * kStreamConsumers < p.V / 4 - pos.step * (kStepEntries / 4)) { a += (double)fa; mn += (double)fm; }
            }
            pos.advance(steps_per_row);
            if (s + 1 < n_steps && pos.row == cur) continue;
            // the end of the row, or of this CTA's run
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); mn += __shfl_xor_sync(0xffffffffu, mn, o); }
            if (lane == 0) { s_a[warp] = a; s_b[warp] = mn; }
            consumers_sync();
            if (warp == 0) {
                a = lane < kStreamWarps ? s_a[lane] : 0.0;
                mn = lane < kStreamWarps ? s_b[lane] : 0.0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); mn += __shfl_xor_sync(0xffffffffu, mn, o); }
                const int share = (int)blockIdx.x - RowShares(cur, steps_per_row, per).first_cta;
                if (lane == 0) {
                    p.slice_abs[row * kTvdSlices + share] = a;
                    p.slice_min[row * kTvdSlices + share] = mn;
                }
            }
            consumers_sync();
            a = 0.0; mn = 0.0;
        }
    }
}

__global__ void tvd_final_kernel(TvdParams p, int steps_per_row, int per) {
    pdl_wait();
    const int rows = p.B * p.gamma, row = blockIdx.x * blockDim.x + threadIdx.x;
    if (row >= rows) return;
    const int n = RowShares(rows - 1 - row, steps_per_row, per).n;
    double a = 0.0, mn = 0.0;
    for (int s = 0; s < n; ++s) { a += p.slice_abs[row * kTvdSlices + s]; mn += p.slice_min[row * kTvdSlices + s]; }
    p.tvd_out[row] = (float)(0.5 * a);
    if (p.accept_prob_out) p.accept_prob_out[row] = (float)mn;
}

// ---------------------------------------------------------------- a row in the shared memory of a cluster
constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kRowMaxCluster = 16;
constexpr int kRowRegGroups = 10;                    // groups of four drafter probabilities a thread holds in registers
constexpr int kRowSlice = kRowRegGroups * 4 * kRowThreads;      // entries per CTA up to which they are all there is
constexpr int kRowMaxSlice = 25 * 1024;              // 100 KB of logits: still two CTAs to an SM

struct RowPublished {
    float m;            // maximum of the slice
    double s;           // sum of exp((z - m) / T) over the slice
    double abs, min;    // the slice's share of the two results
};

// What bounds it: the latency of one pass over a slice and of two exchanges in the cluster, about 10 us.  A CTA puts its
// slice of the logits (cp.async into shared memory) and of the drafter's distribution (registers) in flight at once; one
// exponential per entry, relative to the slice's own maximum.  5 rows of 152,064: 19 us with three kernels, 12 us here.
template <bool STATS_GIVEN>
__global__ void __launch_bounds__(kRowThreads, 3) tvd_row_kernel(TvdParams p, int n_ctas, int slice) {
    extern __shared__ __align__(16) float s_z[];
    __shared__ RowPublished s_pub;
    __shared__ float s_warp_max[kRowWarps];
    __shared__ double s_warp_a[kRowWarps], s_warp_b[kRowWarps];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rank = blockIdx.x % n_ctas, row = blockIdx.x / n_ctas;
    const int v0 = min(p.V, rank * slice), n4 = min(p.V - v0, slice) / 4;         // V and slice are multiples of 4
    float4* z4 = reinterpret_cast<float4*>(s_z);
    pdl_wait();
    pdl_trigger();
    const float4* z = reinterpret_cast<const float4*>(logits_row(p, row) + v0);
    const float4* q = reinterpret_cast<const float4*>(p.draft_probs + (size_t)row * p.V + v0);
    // (a thread reads back the groups it copied itself, so no barrier stands between the copy and its use)
    for (int i = t; i < n4; i += kRowThreads) cp_async_16(&z4[i], z + i);
    float4 qr[kRowRegGroups];
#pragma unroll
    for (int k = 0; k < kRowRegGroups; ++k) {
        const int i = t + k * kRowThreads;
        qr[k] = i < n4 ? __ldcs(q + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");

    float ref, factor;                     // p(v) = exp((z_v - ref) / T) * factor
    if (STATS_GIVEN) {
        // the acceptance scan's merged statistics of logits row b*(gamma+1)+j
        const int b = row / p.gamma, j = row % p.gamma;
        const float2 ms = *reinterpret_cast<const float2*>(p.row_stats + (size_t)(b * (p.gamma + 1) + j) * 2);
        ref = ms.x;
        factor = (float)(1.0 / (double)ms.y);
    } else {
        float m = -INFINITY;
        for (int i = t; i < n4; i += kRowThreads) {
            const float4 x = z4[i];
            m = fmaxf(m, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) s_warp_max[warp] = m;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) m = fmaxf(m, s_warp_max[w]);
        ref = m == -INFINITY ? 0.f : m;    // a slice without a finite logit has weights of zero
        double s = 0.0;
        for (int i = t; i < n4; i += kRowThreads) {
            float4 x = z4[i];
            x.x = expf((x.x - ref) * p.inv_T); x.y = expf((x.y - ref) * p.inv_T);
            x.z = expf((x.z - ref) * p.inv_T); x.w = expf((x.w - ref) * p.inv_T);
            z4[i] = x;
            s += (double)((x.x + x.y) + (x.z + x.w));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) s_warp_a[warp] = s;
        __syncthreads();
        if (t == 0) {
            double total = 0.0;
#pragma unroll
            for (int w = 0; w < kRowWarps; ++w) total += s_warp_a[w];
            s_pub.m = m;
            s_pub.s = total;
        }
        row_barrier(n_ctas);
        // lane r of every warp asks CTA r; a butterfly adds the shares up (the same sum in every lane)
        float mr = -INFINITY;
        double sr = 0.0;
        if (lane < n_ctas) {
            mr = __uint_as_float(peer_load_u32(&s_pub.m, lane));
            sr = __longlong_as_double((long long)peer_load_u64(&s_pub.s, lane));
        }
        float big = mr;
#pragma unroll
        for (int o = kRowMaxCluster / 2; o > 0; o >>= 1) big = fmaxf(big, __shfl_xor_sync(0xffffffffu, big, o));
        big = __shfl_sync(0xffffffffu, big, 0);
        const double scale = lane < n_ctas ? exp(((double)mr - (double)big) * (double)p.inv_T) : 0.0;
        double total = lane < n_ctas ? sr * scale : 0.0;
#pragma unroll
        for (int o = kRowMaxCluster / 2; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        total = __shfl_sync(0xffffffffu, total, 0);
        factor = (float)(__shfl_sync(0xffffffffu, scale, rank) / total);
    }

    double a = 0.0, mn = 0.0;
    auto add = [&](const float4& x, const float4& y) {
        const float e[4] = {x.x, x.y, x.z, x.w}, f[4] = {y.x, y.y, y.z, y.w};
        float fa = 0.f, fm = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float pv = (STATS_GIVEN ? expf((e[i] - ref) * p.inv_T) : e[i]) * factor;
            fa += fabsf(pv - f[i]);
            fm += fminf(pv, f[i]);
        }
        a += (double)fa;
        mn += (double)fm;
    };
#pragma unroll
    for (int k = 0; k < kRowRegGroups; ++k) {
        const int i = t + k * kRowThreads;
        if (i < n4) add(z4[i], qr[k]);
    }
    for (int i0 = t + kRowRegGroups * kRowThreads; i0 < n4; i0 += kRowRegGroups * kRowThreads) {       // slices above kRowSlice
#pragma unroll
        for (int k = 0; k < kRowRegGroups; ++k) { const int i = i0 + k * kRowThreads; if (i < n4) qr[k] = __ldcs(q + i); }
#pragma unroll
        for (int k = 0; k < kRowRegGroups; ++k) { const int i = i0 + k * kRowThreads; if (i < n4) add(z4[i], qr[k]); }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); mn += __shfl_xor_sync(0xffffffffu, mn, o); }
    __syncthreads();                       // s_warp_a has been read
    if (lane == 0) { s_warp_a[warp] = a; s_warp_b[warp] = mn; }
    __syncthreads();
    if (t == 0) {
        a = 0.0; mn = 0.0;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) { a += s_warp_a[w]; mn += s_warp_b[w]; }
        s_pub.abs = a; s_pub.min = mn;
    }
    row_barrier(n_ctas);
    if (rank == 0 && t < 32) {             // CTA 0 adds the shares
        a = 0.0; mn = 0.0;
        if (lane < n_ctas) {
            a = __longlong_as_double((long long)peer_load_u64(&s_pub.abs, lane));
            mn = __longlong_as_double((long long)peer_load_u64(&s_pub.min, lane));
        }
#pragma unroll
        for (int o = kRowMaxCluster / 2; o > 0; o >>= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); mn += __shfl_xor_sync(0xffffffffu, mn, o); }
        if (lane == 0) {
            p.tvd_out[row] = (float)(0.5 * a);
            if (p.accept_prob_out) p.accept_prob_out[row] = (float)mn;
        }
    }
    row_barrier(n_ctas);                   // no CTA leaves while CTA 0 still reads its shared memory
}

// CTAs per row: enough that a slice of the drafter's row fits the registers, more while rows are so few that SMs would
// stay idle (a CTA keeps at least 2,048 entries).
int row_cluster(const TvdParams& p, int rows) {
    int c = 1;
    while (c < kRowMaxCluster && p.V > c * kRowSlice) c *= 2;
    while (c < kRowMaxCluster && (long)rows * c * 2 <= 2 * device_sm_count() && p.V >= 2 * c * 2048) c *= 2;
    return c;
}
// One launch instead of three, as long as the clusters are resident at once: a cluster of many CTAs starts only when
// that many places are free together, and over several waves that costs more than reading the logits twice
// (320 rows of 152,064 in clusters of 16: 144 us).
bool use_row_kernel(const TvdParams& p, int rows) {
    const int c = row_cluster(p, rows);
    return p.V <= kRowMaxSlice * kRowMaxCluster && (c == 1 || (long)rows * c <= 3 * device_sm_count());
}
template <bool STATS_GIVEN>
cudaError_t launch_row(const TvdParams& p, int rows, cudaStream_t stream) {
    const int c = row_cluster(p, rows);
    const int slice = ((p.V + c - 1) / c + 3) / 4 * 4;
    cudaError_t e = cudaFuncSetAttribute(tvd_row_kernel<STATS_GIVEN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kRowMaxSlice * sizeof(float)));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(tvd_row_kernel<STATS_GIVEN>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)(rows * c));
    return c == 1 ? launch_pdl(tvd_row_kernel<STATS_GIVEN>, grid, dim3(kRowThreads), slice * sizeof(float), stream, p, c, slice)
                  : launch_pdl_cluster(tvd_row_kernel<STATS_GIVEN>, grid, dim3(kRowThreads), slice * sizeof(float), stream, c, p, c, slice);
}

}  // namespace

cudaError_t launch_tvd(const TvdParams& p, cudaStream_t stream) {
    const int rows = p.B * p.gamma;
    cudaError_t e = cudaSuccess;
    if (use_row_kernel(p, rows)) {
        e = p.row_stats ? launch_row<true>(p, rows, stream) : launch_row<false>(p, rows, stream);
        if (e != cudaSuccess) return e;
        count_launches(1);
        return cudaGetLastError();
    }
    // Equal runs of the line of steps.  A run is at least a twelfth of a row, so that a row has at most 14 shares (the
    // workspace has room for kTvdSlices).
    const int steps_per_row = (p.V + kStepEntries - 1) / kStepEntries;
    const long total = (long)rows * steps_per_row, sms = device_sm_count();
    if (total > 0x7fffffffL) return cudaErrorInvalidValue;
    const int even = (int)((total + sms - 1) / sms), least = (steps_per_row + 11) / 12;
    const int per = even > least ? even : least;
    const dim3 grid((unsigned)((total + per - 1) / per));
    if (!p.row_stats) {
        e = cudaFuncSetAttribute(tvd_stream_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamSmem);
        if (e == cudaSuccess) e = launch_pdl(tvd_stream_kernel<false>, grid, dim3(kStreamThreads), kStreamSmem, stream, p, steps_per_row, per);
        if (e != cudaSuccess) return e;
        count_launches(1);
    }
    e = cudaFuncSetAttribute(tvd_stream_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStreamSmem);
    if (e == cudaSuccess) e = launch_pdl(tvd_stream_kernel<true>, grid, dim3(kStreamThreads), kStreamSmem, stream, p, steps_per_row, per);
    if (e == cudaSuccess) e = launch_pdl(tvd_final_kernel, dim3((rows + 127) / 128), dim3(128), 0, stream, p, steps_per_row, per);
    if (e != cudaSuccess) return e;
    count_launches(2);
    return cudaGetLastError();
}

}  // namespace massv
