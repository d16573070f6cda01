// Nucleus (top-p) sampling of softmax(z / T), one row per cluster of CTAs (paper Sec. 3.2: the target's
// responses for self-distillation are drawn as sample_top-p(p(. | I, X)); it is also the drafter's sampling
// step when the drafter uses top-p, and probs_out is then the q a verify step needs).
//
// top_p_cluster_kernel keeps the row in the shared memory of 1 .. 8 CTAs, so it crosses HBM once each way;
// top_p_kernel (one CTA per row, the row re-read from L2 by every pass) remains for rows that do not fit there.
//
// Per row: w_v = exp((z_v - max z) / T) in fp32 (ex2.approx), sums in fp64 or in fixed-point integers.  The nucleus - the shortest prefix of the
// tokens ordered by weight (ties: lower index first) whose mass reaches top_p * sum - is found without
// sorting: a search over the bit pattern of w (monotone for non-negative floats) finds the largest
// threshold tau with mass{w >= tau} >= target, which is the weight of the prefix's last token; everything
// above tau is in, and of the tokens equal to tau the first ceil((target - mass{w > tau}) / tau) by index.
// The threshold search is a radix selection in four levels (9 + 9 + 9 + 4 bits of the pattern): each level
// builds a histogram of mass over the next bits of the tokens that match the prefix found so far, and a
// suffix scan over the bins finds the one in which the running mass from the top crosses the target.
// Masses are fixed-point integers there, so the shared-memory atomics add up to the same value whatever
// their order.
// The draw is the inverse CDF in vocabulary order (first index whose running mass exceeds u * total): every
// thread (every warp, in the one-CTA kernel) owns a contiguous range, so the running sums have a fixed order.
#include "kernels.cuh"
#include "ptx.cuh"

namespace massv {

namespace {

constexpr int kTopPThreads = 1024;
constexpr int kTopPWarps = kTopPThreads / 32;

// Integer versions (exact, so any order gives the same value).
__device__ __forceinline__ unsigned long long block_sum_u64(unsigned long long x, unsigned long long* sm) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sm[warp] = x;
    __syncthreads();
    unsigned long long s = 0ull;
#pragma unroll
    for (int w = 0; w < kTopPWarps; ++w) s += sm[w];
    return s;
}
// Sum of the values of all threads with a higher index.
__device__ __forceinline__ unsigned long long block_suffix_exclusive_u64(unsigned long long x, unsigned long long* sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_down_sync(0xffffffffu, incl, o);
        if (lane + o < 32) incl += y;
    }
    __syncthreads();
    if (lane == 0) sm[warp] = incl;
    __syncthreads();
    unsigned long long above = 0ull;
#pragma unroll
    for (int w = 0; w < kTopPWarps; ++w) if (w > warp) above += sm[w];
    return above + incl - x;
}

// w = 2^((z - max) * log2(e) / T): one multiply-add into the exponential unit.  Every pass of a kernel uses this
// same function, so thresholds, ties and sums are consistent with one another.
struct RowWeight {
    float k2, m2;
    __device__ RowWeight(float inv_T, float m) : k2(inv_T * 1.4426950408889634f) { m2 = -m * k2; }
    __device__ __forceinline__ float operator()(float zv) const {
        return fminf(ex2_ftz(fmaf(zv, k2, m2)), 1.0f);              // the approximation must not step past the pattern of 1.0f
    }
};
// The mass that the nucleus must reach, of a row of `total` units.  (top_p = 1 is the whole row as it stands: totals from 2^53 up - rows whose
// weights add up to more than 512 - lose low bits as a double, and with them entries of the tail.)
__device__ __forceinline__ unsigned long long target_mass(float top_p, unsigned long long total) {
    if (top_p >= 1.f) return total;
    const unsigned long long target = (unsigned long long)ceil((double)top_p * (double)total);
    return min(max(target, 1ull), total);
}
// floor(w * 2^fx_bits) for 0 <= w <= 1 from the pattern of w: mantissa shifted by the exponent
__device__ __forceinline__ unsigned long long fixed_point(float w, int fx_bits) {
    const uint32_t b = __float_as_uint(w);
    const int e = (int)(b >> 23);                      // biased exponent; 0 = zero (denormals are flushed)
    if (e == 0) return 0ull;
    const unsigned long long mant = (unsigned long long)((b & 0x7FFFFFu) | 0x800000u);
    const int sh = e - 127 - 23 + fx_bits;             // w = mant * 2^(e - 127 - 23)
    return sh >= 0 ? mant << sh : (sh > -24 ? mant >> (-sh) : 0ull);
}
// the same number for fx_bits = 44 as two 32-bit words, from two float -> integer conversions:
// hi = floor(w * 2^12), lo = floor((w - hi * 2^-12) * 2^44); both products and the difference are exact
__device__ __forceinline__ void fixed_words_44(float w, uint32_t& hi, uint32_t& lo) {
    hi = __float2uint_rz(w * 4096.f);
    lo = __float2uint_rz(fmaf(-(float)hi, 1.f / 4096.f, w) * 17592186044416.f);
}

constexpr int kTopPBins = 512;      // 9 bits of the pattern per level (9 + 9 + 9 + 4)
constexpr int kTopPCopies = 8;
constexpr int kTopPMaxBlocks = kTopPBins * kTopPCopies / kTopPWarps;     // 512-entry blocks per warp: 128, i.e. V <= 2^21

__global__ void __launch_bounds__(kTopPThreads) top_p_kernel(TopPParams p) {
    const int row = blockIdx.x, t = threadIdx.x;
    const float* z = p.logits + (size_t)row * p.V;
    // 32 KB used twice: the histograms' low and high words during the threshold search, then the masses
    // of the 512-entry blocks of every warp's range
    __shared__ __align__(16) unsigned long long pool[kTopPBins * kTopPCopies];
    uint32_t* hist_lo = reinterpret_cast<uint32_t*>(pool);
    uint32_t* hist_hi = hist_lo + kTopPBins * kTopPCopies;
    double* block_mass = reinterpret_cast<double*>(pool);          // [kTopPWarps][kTopPMaxBlocks]
    __shared__ unsigned long long sm_u64[kTopPWarps];
    __shared__ int s_bin;
    __shared__ unsigned long long s_above;
    __shared__ float sm_max[kTopPWarps];
    __shared__ int s_first, s_last;
    pdl_wait();
    pdl_trigger();

    // Every pass walks the row with sixteen independent loads in flight per thread (the row comes from L2,
    // a few hundred cycles away); entries past the end read as -inf, whose weight is zero.
    constexpr int kUnroll = 16;
    auto load4 = [&](int v_first, int stride, float (&zz)[kUnroll]) {
#pragma unroll
        for (int j = 0; j < kUnroll; ++j) { const int v = v_first + j * stride; zz[j] = v < p.V ? z[v] : -INFINITY; }
    };

    // ---- row maximum
    float m = -INFINITY;
    for (int v = t; v < p.V; v += kUnroll * kTopPThreads) {
        float zz[kUnroll];
        load4(v, kTopPThreads, zz);
#pragma unroll
        for (int j = 0; j < kUnroll; ++j) m = fmaxf(m, zz[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((t & 31) == 0) sm_max[t >> 5] = m;
    __syncthreads();
    m = sm_max[0];
#pragma unroll
    for (int w = 1; w < kTopPWarps; ++w) m = fmaxf(m, sm_max[w]);
    if (!(m > -INFINITY) || !(m < INFINITY)) {          // no finite logit in the row: nothing to draw from
        if (t == 0) { p.tokens[row] = 0; set_status(p.dev_status, MASSV_ERR_INVALID_ARG); }
        return;
    }
    const RowWeight weight_of(p.inv_T, m);

    // ---- total mass, in fixed point: w * 2^fx_bits truncated; the row's sum stays below 2^63 for V <= 2^19
    const int fx_bits = p.V <= (1 << 19) ? 44 : 30;
    auto fixed_words = [&](float w, uint32_t& hi, uint32_t& lo) {
        if (fx_bits == 44) {
            fixed_words_44(w, hi, lo);
        } else {
            const unsigned long long f = fixed_point(w, fx_bits);
            hi = (uint32_t)(f >> 32); lo = (uint32_t)f;
        }
    };
    unsigned long long local_hi = 0ull, local_lo = 0ull;
    for (int v = t; v < p.V; v += kUnroll * kTopPThreads) {
        float zz[kUnroll];
        load4(v, kTopPThreads, zz);
#pragma unroll
        for (int j = 0; j < kUnroll; ++j) {
            uint32_t hi, lo;
            fixed_words(weight_of(zz[j]), hi, lo);
            local_hi += hi; local_lo += lo;
        }
    }
    const unsigned long long S_fx = (block_sum_u64(local_hi, sm_u64) << 32) + block_sum_u64(local_lo, sm_u64);
    const unsigned long long target_fx = target_mass(p.top_p, S_fx);

    // ---- threshold: largest bit pattern tau with mass{w >= tau} >= target, by radix selection
    uint32_t prefix = 0u;                 // bits of tau found so far
    unsigned long long mass_above = 0ull; // mass of the tokens whose pattern is above every pattern with this prefix
#pragma unroll
    for (int level = 0; level < 4; ++level) {
        const int shift = level == 0 ? 22 : (level == 1 ? 13 : (level == 2 ? 4 : 0));
        const int bits = level == 3 ? 4 : 9, nbins = 1 << bits;
        const uint32_t hi_mask = level == 0 ? 0u : ~((1u << (shift + bits)) - 1u);       // bits already fixed
        for (int i = t; i < kTopPBins * kTopPCopies; i += kTopPThreads) { hist_lo[i] = 0u; hist_hi[i] = 0u; }
        __syncthreads();
        // many tokens share their leading bits: eight copies of the histogram, chosen by lane, keep
        // the atomics on a hot bin from queueing behind one another
        // (64-bit sums as two 32-bit words with an explicit carry: 32-bit shared-memory atomics are native)
        const int my_copy = (t & (kTopPCopies - 1)) * kTopPBins;
        for (int v = t; v < p.V; v += kUnroll * kTopPThreads) {
            float zz[kUnroll];
            load4(v, kTopPThreads, zz);
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const float w = weight_of(zz[j]);
                const uint32_t b = __float_as_uint(w);
                if ((b & hi_mask) == prefix) {
                    uint32_t hi, lo;
                    fixed_words(w, hi, lo);
                    const int bin = my_copy + (int)((b >> shift) & (uint32_t)(nbins - 1));
                    if (lo) hi += (atomicAdd(&hist_lo[bin], lo) > ~lo) ? 1u : 0u;      // the low word wrapped
                    if (hi) atomicAdd(&hist_hi[bin], hi);
                }
            }
        }
        __syncthreads();
        // suffix sums over the bins, highest first: thread t < 512 owns bin t (all copies)
        unsigned long long own = 0ull;
        if (t < nbins) {
#pragma unroll
            for (int c = 0; c < kTopPCopies; ++c)
                own += ((unsigned long long)hist_hi[c * kTopPBins + t] << 32) + (unsigned long long)hist_lo[c * kTopPBins + t];
        }
        const unsigned long long above_me = block_suffix_exclusive_u64(own, sm_u64);        // mass in bins above t
        // the bin b with mass_above + sum(bins > b) < target <= mass_above + sum(bins >= b) exists exactly once
        const unsigned long long run = mass_above + above_me;
        if (run < target_fx && run + own >= target_fx) { s_bin = t; s_above = run; }
        __syncthreads();
        prefix |= (uint32_t)s_bin << shift;
        mass_above = s_above;
        __syncthreads();
    }
    const uint32_t tau = prefix;
    // how many of the tokens equal to tau the prefix takes (at least one: mass{w > tau} < target)
    const unsigned long long tau_fx = fixed_point(__uint_as_float(tau), fx_bits);
    unsigned long long n_ties_u = tau_fx ? (target_fx - mass_above + tau_fx - 1ull) / tau_fx : ~0ull;
    if (n_ties_u < 1ull) n_ties_u = 1ull;
    const long long n_ties = n_ties_u > (unsigned long long)4e18 ? (long long)4e18 : (long long)n_ties_u;

    // ---- ordered passes: warp w owns a contiguous range, walked 32 consecutive entries at a time
    // (lane = entry, so loads and stores are coalesced); ranks among the entries equal to tau come
    // from ballots, running masses from warp-wide sums in round order.
    const int warp = t >> 5, lane = t & 31;
    const int per_warp = ((p.V + kTopPWarps - 1) / kTopPWarps + 31) / 32 * 32;
    const int w0 = min(p.V, warp * per_warp), w1 = min(p.V, w0 + per_warp);
    const unsigned lt_mask = (1u << lane) - 1u;
    __shared__ long long warp_ties[kTopPWarps];
    __shared__ double warp_mass[kTopPWarps];
    // ties per warp
    {
        long long n = 0;
        for (int v = w0 + lane; v - lane < w1; v += kUnroll * 32) {
            float zz[kUnroll];
            load4(v, 32, zz);
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const bool tie = (v + j * 32 < w1) && __float_as_uint(weight_of(zz[j])) == tau;
                n += __popc(__ballot_sync(0xffffffffu, tie));
            }
        }
        if (lane == 0) warp_ties[warp] = n;
    }
    __syncthreads();
    long long tie_base = 0;
    for (int w = 0; w < warp; ++w) tie_base += warp_ties[w];
    // mass per warp (members only): per block of 16 rounds (512 entries) every lane adds up its own
    // entries, then one warp-wide sum; the block masses are kept for the draw
    __syncthreads();                             // the histograms are not read any more: the pool changes hands
    {
        long long rank0 = tie_base;              // ties before the current round
        double acc = 0.0;
        int blk = 0;
        for (int v = w0 + lane; v - lane < w1; v += kUnroll * 32, ++blk) {
            float zz[kUnroll];
            load4(v, 32, zz);
            double x = 0.0;
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const float w = (v + j * 32 < w1) ? weight_of(zz[j]) : 0.f;
                const uint32_t b = __float_as_uint(w);
                const bool tie = (v + j * 32 < w1) && b == tau;
                const unsigned ties = __ballot_sync(0xffffffffu, tie);
                const bool in = (v + j * 32 < w1) && (b > tau || (tie && rank0 + __popc(ties & lt_mask) < n_ties));
                rank0 += __popc(ties);
                if (in) x += (double)w;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) block_mass[warp * kTopPMaxBlocks + blk] = x;
            acc += x;
        }
        if (lane == 0) warp_mass[warp] = acc;
    }
    __syncthreads();
    double Z = 0.0, base = 0.0;
    for (int w = 0; w < kTopPWarps; ++w) { if (w < warp) base += warp_mass[w]; Z += warp_mass[w]; }
    const double target = (double)p.u[row] * Z;
    // the warp whose range holds the target walks it again with running sums; the last warp with mass
    // keeps the fall-back (rounding can push the target past the end)
    if (t == 0) { s_first = 0x7fffffff; s_last = -1; }
    __syncthreads();
    const bool holds = warp_mass[warp] > 0.0 && base <= target && target < base + warp_mass[warp];
    bool last_with_mass = warp_mass[warp] > 0.0;
    for (int w = warp + 1; w < kTopPWarps; ++w) last_with_mass = last_with_mass && !(warp_mass[w] > 0.0);
    const float inv_Z = (float)(1.0 / Z);
    {
        long long rank0 = tie_base;
        double run = base;                       // mass before the current block / round
        int first = 0x7fffffff, last = -1;
        int blk = 0;
        for (int v = w0 + lane; v - lane < w1; v += kUnroll * 32, ++blk) {
            float zz[kUnroll];
            load4(v, 32, zz);
            // only the block that holds the target is walked round by round with running sums
            const double blk_mass = block_mass[warp * kTopPMaxBlocks + blk];
            const bool scan = holds && first == 0x7fffffff && blk_mass > 0.0 && run <= target && target < run + blk_mass;
            double run_in = run;
            int blk_last = -1;
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const int vv = v + j * 32;
                const float w = vv < w1 ? weight_of(zz[j]) : 0.f;
                const uint32_t b = __float_as_uint(w);
                const bool tie = vv < w1 && b == tau;
                const unsigned ties = __ballot_sync(0xffffffffu, tie);
                const bool in = vv < w1 && w > 0.f && (b > tau || (tie && rank0 + __popc(ties & lt_mask) < n_ties));
                rank0 += __popc(ties);
                if (p.probs_out && vv < w1) p.probs_out[(size_t)row * p.V + vv] = in ? w * inv_Z : 0.f;
                if (in) { last = vv; blk_last = vv; }
                if (scan) {
                    // inclusive sum over the lanes of this round, in lane order
                    double incl = in ? (double)w : 0.0;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const double y = __shfl_up_sync(0xffffffffu, incl, o);
                        if (lane >= o) incl += y;
                    }
                    if (in && first == 0x7fffffff && run_in + incl > target) first = vv;
                    run_in += __shfl_sync(0xffffffffu, incl, 31);
                }
            }
            if (scan) {
                // (the round sums and the block's mass add the same numbers in another order: if the last bit
                // puts the target past the running sum, the block's last member is the answer)
                first = __reduce_min_sync(0xffffffffu, first);
                if (first == 0x7fffffff) first = __reduce_max_sync(0xffffffffu, blk_last);
            }
            run += blk_mass;
        }
        first = __reduce_min_sync(0xffffffffu, first);
        last = __reduce_max_sync(0xffffffffu, last);
        if (holds && first == 0x7fffffff && last >= 0) first = last;      // no block claimed the target (rounding): the warp's last member
        if (holds && first != 0x7fffffff) atomicMin(&s_first, first);
        if (last_with_mass && last >= 0) atomicMax(&s_last, last);
    }
    __syncthreads();
    if (t == 0) p.tokens[row] = s_first != 0x7fffffff ? s_first : s_last;      // rounding past the end: last nucleus token
}

// ---------------------------------------------------------------- a row in the shared memory of a cluster
constexpr int kRowThreads = 512;
constexpr int kRowWarps = kRowThreads / 32;
constexpr int kRowCopies = 4;                        // copies of a histogram, chosen by lane
constexpr int kRowCopyStride = kTopPBins + 8;        // the copies of a bin lie in different banks
constexpr int kRowMaxCluster = 8;
constexpr int kRowCand = 32;                         // candidates for tau that a CTA can publish
// Entries per CTA: up to kRowPairSlice two CTAs share an SM (one works while the other waits for its row or for a
// barrier of its cluster); up to kRowMaxSlice the slice still fits.
constexpr int kRowPairSlice = 21 * 1024;
constexpr int kRowMaxSlice = 48 * 1024;
static_assert(kRowThreads == kTopPBins && kRowThreads >= kRowMaxCluster * kRowCand, "one thread per bin, one per candidate");
static_assert(kRowMaxSlice * kRowMaxCluster <= (1 << 19), "fixed point with 44 bits");

// What a CTA lets the rest of its cluster read.
struct RowPublished {
    unsigned long long hist[2][kTopPBins];   // two levels of the threshold search take turns
    unsigned long long max_bits;
    unsigned long long mass;                 // bits of a double: mass above the candidates (later: above tau)
    unsigned long long n_cand;               // entries that share the bits of tau found by then
    uint32_t cand[kRowCand];                 // their patterns, in no particular order
};

// What bounds it: the row crosses HBM once in and once out (8 B per entry); between the two lie three barriers of the
// cluster (about 2 us each with the exchange behind them) and three walks over the slice in shared memory (1 - 3.5 us
// with two CTAs on an SM), a serial chain of about 22 us per CTA.  64 rows of 152,064 with probs_out: 188 us with one CTA
// per row re-reading it from L2 in nine passes (64 of 148 SMs busy), 54 us here (two waves of CTAs).
__global__ void __launch_bounds__(kRowThreads, 2) top_p_cluster_kernel(TopPParams p, int n_ctas, int slice) {
    extern __shared__ __align__(16) float s_w[];                 // the slice: logits, then weights
    __shared__ uint32_t hist_lo[kRowCopies * kRowCopyStride], hist_hi[kRowCopies * kRowCopyStride];
    __shared__ RowPublished s_pub;
    __shared__ unsigned long long s_warp[kRowWarps], s_warp_light[kRowWarps];
    __shared__ double s_warp_mass[kRowWarps];
    __shared__ int s_warp_ties[kRowWarps];
    __shared__ float s_warp_max[kRowWarps];
    __shared__ uint32_t s_cand[kRowMaxCluster * kRowCand], s_tau;
    __shared__ double s_cta_mass[kRowMaxCluster], s_cand_mass[kRowMaxCluster];
    __shared__ int s_cta_count[kRowMaxCluster], s_cand_ties[kRowMaxCluster];
    __shared__ unsigned long long s_above;
    __shared__ int s_bin, s_in_bin, s_n_cand, s_owner, s_owner_last;

    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int rank = blockIdx.x % n_ctas, row = blockIdx.x / n_ctas;
    const int v0 = min(p.V, rank * slice), n = min(p.V - v0, slice), n4 = (n + 3) / 4;
    const float* z = p.logits + (size_t)row * p.V + v0;
    for (int i = t; i < kRowCopies * kRowCopyStride; i += kRowThreads) { hist_lo[i] = 0u; hist_hi[i] = 0u; }
    if (t == 0) { s_owner = 0x7fffffff; s_owner_last = -1; s_n_cand = 0; }
    pdl_wait();
    pdl_trigger();

    // ---- the slice into shared memory, its maximum on the way; the last group of four is padded with -inf
    float m = -INFINITY;
    if (((reinterpret_cast<uintptr_t>(z) & 15u) == 0) && n % 4 == 0) {
        constexpr int kUnroll = 8;                               // 16-byte loads in flight per thread
        for (int i = t; i < n4; i += kUnroll * kRowThreads) {
            float4 x[kUnroll];
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const int k = i + j * kRowThreads;
                x[j] = k < n4 ? __ldcs(reinterpret_cast<const float4*>(z) + k) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
            }
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const int k = i + j * kRowThreads;
                if (k < n4) reinterpret_cast<float4*>(s_w)[k] = x[j];
                m = fmaxf(m, fmaxf(fmaxf(x[j].x, x[j].y), fmaxf(x[j].z, x[j].w)));
            }
        }
    } else {
        constexpr int kUnroll = 16;
        for (int i = t; i < 4 * n4; i += kUnroll * kRowThreads) {
            float x[kUnroll];
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) { const int k = i + j * kRowThreads; x[j] = k < n ? __ldcs(z + k) : -INFINITY; }
#pragma unroll
            for (int j = 0; j < kUnroll; ++j) {
                const int k = i + j * kRowThreads;
                if (k < 4 * n4) s_w[k] = x[j];
                m = fmaxf(m, x[j]);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) s_warp_max[warp] = m;
    __syncthreads();
    m = s_warp_max[0];
#pragma unroll
    for (int w = 1; w < kRowWarps; ++w) m = fmaxf(m, s_warp_max[w]);
    if (n_ctas > 1) {
        if (t == 0) s_pub.max_bits = (unsigned long long)__float_as_uint(m);
        row_barrier(n_ctas);
        // (lane r of every warp asks CTA r)
        if (lane < n_ctas) m = fmaxf(m, __uint_as_float((uint32_t)peer_load_u64(&s_pub.max_bits, lane)));
#pragma unroll
        for (int o = kRowMaxCluster / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        m = __shfl_sync(0xffffffffu, m, 0);
    }
    if (!(m > -INFINITY) || !(m < INFINITY)) {          // no finite logit in the row: nothing to draw from
        if (rank == 0 && t == 0) { p.tokens[row] = 0; set_status(p.dev_status, MASSV_ERR_INVALID_ARG); }
        row_barrier(n_ctas);                            // no CTA leaves while another still reads its shared memory
        return;
    }
    const RowWeight weight_of(p.inv_T, m);

    // ---- threshold: largest bit pattern tau with mass{w >= tau} >= target, by radix selection: a first level of 32 bins per
    // power of two, levels of 9 bits more while more than kRowCand entries share the bits found, then those entries one by
    // one.  A bin fixes the exponent, so its mass is a sum of (truncated) mantissas: a word that wraps every 256 entries at
    // most, and a carry.  A language model's row needs the first level only; with two bins per power of two it took a second
    // walk and exchange (64 rows of 152,064: 61 us, 53 here).  Rows with more entries near the threshold take the second level here too, and
    // reading 385 bins of every peer instead of 26 shows (logits of standard deviation 2.5, one row of 152,064: 30.5 us, 32.0 here).
    uint32_t prefix = 0u;                 // bits of tau found so far: all but the last `open` ones
    int open = 0;
    unsigned long long mass_above = 0ull, target_fx = 0ull, total_fx = 0ull;
    const int my_copy = (lane & (kRowCopies - 1)) * kRowCopyStride;
    auto mantissa = [&](uint32_t b) { return ((b & 0x7FFFFFu) | 0x800000u) >> min(max(106 - (int)(b >> 23), 0), 31); };      // zero below 2^-44
    // four entries at a time, so that four atomics are in flight before the first result is looked at
    auto add4 = [&](const uint32_t (&v)[4], const int (&bin)[4]) {
        uint32_t old[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) { old[j] = 0u; if (v[j]) old[j] = atomicAdd(&hist_lo[my_copy + bin[j]], v[j]); }
#pragma unroll
        for (int j = 0; j < 4; ++j) if (old[j] > ~v[j]) atomicAdd(&hist_hi[my_copy + bin[j]], 1u);      // the word wrapped
    };
    // One level once the copies are filled: the cluster's bins, and the one in which the running mass from the top
    // crosses the target.  Bin t < n_bins stands for the patterns from `low` + (t << shift) on; bin sum_bin, if the level
    // has one, is the sum of the light entries (in units of 2^-44).
    int half = 0;                         // which of the two published histograms is next
    auto find_bin = [&](uint32_t low, int shift, int n_bins, int sum_bin) {
        __syncthreads();
        // thread t owns bin t: its copies, cleared for the next level, then the other CTAs' share of it
        unsigned long long own = 0ull;
#pragma unroll
        for (int c = 0; c < kRowCopies; ++c) {
            const int at = c * kRowCopyStride + t;
            own += ((unsigned long long)hist_hi[at] << 32) + (unsigned long long)hist_lo[at];
            hist_hi[at] = 0u; hist_lo[at] = 0u;
        }
        if (t == sum_bin) {
            own = 0ull;
#pragma unroll
            for (int w = 0; w < kRowWarps; ++w) own += s_warp_light[w];
        }
        if (n_ctas > 1) {
            s_pub.hist[half][t] = own;
            // (a CTA writes this half again two levels on: every CTA has then passed the next level's barrier,
            // which it reaches after these reads)
            row_barrier(n_ctas);
            own = 0ull;
            if (t < n_bins || t == sum_bin) {
                unsigned long long part[kRowMaxCluster];
#pragma unroll
                for (int r = 0; r < kRowMaxCluster; ++r) part[r] = r < n_ctas ? peer_load_u64(&s_pub.hist[half][t], r) : 0ull;
#pragma unroll
                for (int r = 0; r < kRowMaxCluster; ++r) own += part[r];
            }
        }
        // mantissas -> units of 2^-44
        const uint32_t bits = low + ((uint32_t)t << shift);
        const unsigned long long in_units = t == sum_bin ? own : own << max((int)(bits >> 23) - 106, 0);
        // suffix sums over the bins, highest first (the light entries below all others)
        unsigned long long incl = t == sum_bin ? 0ull : in_units;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long y = __shfl_down_sync(0xffffffffu, incl, o);
            if (lane + o < 32) incl += y;
        }
        if (lane == 0) s_warp[warp] = incl;
        if (t == sum_bin) s_above = in_units;
        __syncthreads();
        unsigned long long above = 0ull, total = 0ull;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) { total += s_warp[w]; if (w > warp) above += s_warp[w]; }
        unsigned long long run = mass_above + above + incl - in_units;
        if (sum_bin >= 0) {
            if (t == sum_bin) run = total;
            total += s_above;
            total_fx = total;
            target_fx = target_mass(p.top_p, total);
            __syncthreads();                       // s_above has been read
        }
        // the bin b with mass_above + sum(bins > b) < target <= mass_above + sum(bins >= b) exists exactly once
        if (run < target_fx && run + in_units >= target_fx) {
            s_bin = t;
            s_above = run;
            // entries in the bin, at most: none is lighter than the bin's lower end
            const unsigned long long most = own / max(1u, mantissa(bits));
            s_in_bin = most < 0x7fffffffull ? (int)most : 0x7fffffff;
        }
        __syncthreads();
        const bool among_light = s_bin == sum_bin;
        prefix = among_light ? 0u : low + ((uint32_t)s_bin << shift);
        open = shift;
        mass_above = s_above;
        half ^= 1;
    };
    // All groups of four entries whose largest is at least `from` (the others hold nothing of interest: one comparison).
    auto walk = [&](uint32_t from_bits, auto&& f) {
        const float from = __uint_as_float(from_bits);
        for (int i = t; i < n4; i += 2 * kRowThreads) {
            const int i2 = i + kRowThreads;
            const float4 x = reinterpret_cast<const float4*>(s_w)[i];
            const float4 y = i2 < n4 ? reinterpret_cast<const float4*>(s_w)[i2] : make_float4(0.f, 0.f, 0.f, 0.f);
            if (fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)) >= from) f(x);
            if (fmaxf(fmaxf(y.x, y.y), fmaxf(y.z, y.w)) >= from) f(y);          // (from > 0)
        }
    };
    auto add_matching = [&](int shift) {       // histogram of the entries that share the bits found so far, by the bits from `shift` on
        const uint32_t from = prefix;
        const int known = open;
        walk(from, [&](const float4& x) {
            const uint32_t b[4] = {__float_as_uint(x.x), __float_as_uint(x.y), __float_as_uint(x.z), __float_as_uint(x.w)};
            uint32_t v[4];
            int bin[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) { v[j] = (b[j] >> known) == (from >> known) ? mantissa(b[j]) : 0u; bin[j] = (int)((b[j] - from) >> shift); }
            add4(v, bin);
        });
    };
    // The first level turns the logits into weights on the way.  Most entries of a row are light (below 2^-12 of the
    // largest), and tau rarely is: they go into one sum in registers instead of the histogram, which is what the walk
    // waits for (64 rows of 152,064, logits of standard deviation 5: 5.3 -> 3.5 us).  If tau lies among them after all,
    // another walk counts them.
    constexpr uint32_t kLightBits = 115u << 23;         // 2^-12
    unsigned long long light = 0ull;
    for (int i = t; i < n4; i += kRowThreads) {
        float4 x = reinterpret_cast<const float4*>(s_w)[i];
        x = make_float4(weight_of(x.x), weight_of(x.y), weight_of(x.z), weight_of(x.w));
        reinterpret_cast<float4*>(s_w)[i] = x;
        const uint32_t b[4] = {__float_as_uint(x.x), __float_as_uint(x.y), __float_as_uint(x.z), __float_as_uint(x.w)};
        uint32_t v[4];
        int bin[4];
        bool heavy = false;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const bool h = b[j] >= kLightBits;
            heavy = heavy || h;
            v[j] = h ? mantissa(b[j]) : 0u;
            bin[j] = (int)((b[j] - kLightBits) >> 18);
            // floor(w * 2^44) < 2^32: the mantissa in the word's upper 24 bits, shifted down (shr gives zero from 32 on)
            uint32_t f;
            asm("shr.u32 %0, %1, %2;" : "=r"(f) : "r"(((b[j] & 0x7FFFFFu) | 0x800000u) << 8), "r"(114u - (b[j] >> 23)));
            light += h ? 0u : f;
        }
        if (heavy) add4(v, bin);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) light += __shfl_xor_sync(0xffffffffu, light, o);
    if (lane == 0) s_warp_light[warp] = light;
    find_bin(kLightBits, 18, 12 * 32 + 1, kRowThreads - 1);          // (2^-12 <= w <= 1; the last bin is free for the light sum)
    auto publish = [&](double mass, int count) {           // this CTA's mass and count, visible to the cluster on return
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) { mass += __shfl_xor_sync(0xffffffffu, mass, o); count += __shfl_xor_sync(0xffffffffu, count, o); }
        if (lane == 0) { s_warp_mass[warp] = mass; s_warp_ties[warp] = count; }
        __syncthreads();
        if (warp == 0) {
            double a = lane < kRowWarps ? s_warp_mass[lane] : 0.0;
            int c = lane < kRowWarps ? s_warp_ties[lane] : 0;
#pragma unroll
            for (int o = kRowWarps / 2; o > 0; o >>= 1) { a += __shfl_xor_sync(0xffffffffu, a, o); c += __shfl_xor_sync(0xffffffffu, c, o); }
            if (lane == 0) { s_pub.mass = (unsigned long long)__double_as_longlong(a); s_pub.n_cand = (unsigned long long)c; }
        }
        row_barrier(n_ctas);
    };
    constexpr uint32_t kLowest = 83u << 23;       // 2^-44: lighter entries have no mass
    // What the last walk leaves: every CTA's mass above tau and the number of entries that may be tau (listed: which they are).
    double mass_gt = 0.0;
    int n_equal = 0;
    const bool everything = target_fx == total_fx;        // the same in all CTAs
    bool listed = false;
    if (everything) {
        // top_p takes the whole row: tau is the lightest entry that has mass
        uint32_t least = 0xffffffffu;
        walk(kLowest, [&](const float4& x) {
            const float w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t b = __float_as_uint(w[j]);
                if (b >= kLowest) {
                    mass_gt += (double)w[j];
                    n_equal = b < least ? 1 : n_equal + (b == least ? 1 : 0);
                    least = min(least, b);
                }
            }
        });
        const uint32_t warp_least = __reduce_min_sync(0xffffffffu, least);
        if (lane == 0) s_cand[warp] = warp_least;
        __syncthreads();
        uint32_t cta_least = s_cand[0];
#pragma unroll
        for (int w = 1; w < kRowWarps; ++w) cta_least = min(cta_least, s_cand[w]);
        if (least != cta_least) n_equal = 0;
        if (t < kRowCand) s_pub.cand[t] = cta_least;
    } else {
        if (prefix == 0u) {                       // the crossing lies among the light entries (same in all CTAs)
            walk(1u, [&](const float4& x) {
                const uint32_t b[4] = {__float_as_uint(x.x), __float_as_uint(x.y), __float_as_uint(x.z), __float_as_uint(x.w)};
                uint32_t v[4];
                int bin[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) { v[j] = b[j] < kLightBits ? mantissa(b[j]) : 0u; bin[j] = (int)((b[j] - kLowest) >> 19); }
                add4(v, bin);
            });
            find_bin(kLowest, 19, kTopPBins, -1); // 2^-44 <= w < 2^-12, 16 bins per power of two
        }
        while (open > 0 && s_in_bin > kRowCand) {
            const int shift = max(open - 9, 0);
            add_matching(shift);
            find_bin(prefix, shift, 1 << (open - shift), -1);
        }

        // ---- Few entries share the bits of tau found so far (or all of it is known): every CTA adds up what lies above and
        // publishes the candidates, and the whole cluster resolves tau, the ties and the masses from one exchange.
        const uint32_t lead = prefix >> open;
        const int known = open;
        listed = s_in_bin <= kRowCand;            // (then the candidates of all CTAs together fit one list)
        walk(prefix, [&](const float4& x) {
            const float w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t b = __float_as_uint(w[j]);
                if ((b >> known) > lead) mass_gt += (double)w[j];
                else if ((b >> known) == lead) {
                    ++n_equal;
                    if (listed) {
                        const int k = atomicAdd(&s_n_cand, 1);
                        if (k < kRowCand) s_pub.cand[k] = b;
                    }
                }
            }
        });
    }
    publish(mass_gt, n_equal);
    // warp r asks CTA r: its mass, its count, and one candidate per lane
    uint32_t c = 0u;
    if (warp < kRowMaxCluster) {
        const int asked = min(warp, n_ctas - 1);
        const uint32_t theirs = peer_load_u32(&s_pub.cand[lane], asked);
        const unsigned long long mass = peer_load_u64(&s_pub.mass, asked), count = peer_load_u64(&s_pub.n_cand, asked);
        if (everything ? warp < n_ctas : (listed && warp < n_ctas && lane < (int)count)) c = theirs;
        s_cand[t] = c;
        if (lane == 0) {
            s_cta_mass[warp] = warp < n_ctas ? __longlong_as_double((long long)mass) : 0.0;
            s_cta_count[warp] = warp < n_ctas ? (int)count : 0;
        }
    }
    __syncthreads();
    double mass_of[kRowMaxCluster];                        // mass above tau, later of the members, of every CTA
    int n_of[kRowMaxCluster];                              // candidates, later ties, of every CTA
#pragma unroll
    for (int r = 0; r < kRowMaxCluster; ++r) { mass_of[r] = s_cta_mass[r]; n_of[r] = s_cta_count[r]; }
    float tau = __uint_as_float(prefix);          // more entries than a list holds share every bit: it is tau, and they are the ties
    if (everything) {
        uint32_t least = 0xffffffffu;
#pragma unroll
        for (int r = 0; r < kRowMaxCluster; ++r) if (r < n_ctas) least = min(least, s_cand[r * kRowCand]);
        tau = __uint_as_float(least);
        const unsigned long long tau_fx = (unsigned long long)mantissa(least) << max((int)(least >> 23) - 106, 0);
        unsigned long long ties_fx = 0ull;
#pragma unroll
        for (int r = 0; r < kRowMaxCluster; ++r) {
            if (s_cand[r * kRowCand] != least) n_of[r] = 0;
            mass_of[r] -= (double)n_of[r] * (double)tau;
            ties_fx += (unsigned long long)n_of[r] * tau_fx;
        }
        mass_above = target_fx - ties_fx;
    } else if (listed) {
        if (c != 0u) {
            // the candidate at which the running mass from the top crosses the target is tau (all have one exponent)
            unsigned long long gt = 0ull, eq = 0ull;
#pragma unroll
            for (int r = 0; r < kRowMaxCluster; ++r)
                for (int j = 0; j < n_of[r]; ++j) {
                    const uint32_t o = s_cand[r * kRowCand + j], f = mantissa(o);
                    gt += o > c ? f : 0u;
                    eq += o == c ? f : 0u;
                }
            const int up = max((int)(c >> 23) - 106, 0);
            gt = mass_above + (gt << up);
            if (gt < target_fx && gt + (eq << up) >= target_fx) { s_tau = c; s_above = gt; }
        }
        __syncthreads();
        tau = __uint_as_float(s_tau);
        mass_above = s_above;
        if (warp < kRowMaxCluster) {
            // (one exponent, at most 32 terms of 24 bits: the sum is exact whatever the order of the list)
            double above = __uint_as_float(c) > tau ? (double)__uint_as_float(c) : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) above += __shfl_xor_sync(0xffffffffu, above, o);
            const unsigned eq = __ballot_sync(0xffffffffu, __uint_as_float(c) == tau);
            if (lane == 0) { s_cand_mass[warp] = above; s_cand_ties[warp] = __popc(eq); }
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kRowMaxCluster; ++r) { mass_of[r] += s_cand_mass[r]; n_of[r] = s_cand_ties[r]; }
    }
    if (n_ctas > 1) asm volatile("barrier.cluster.arrive.release;" ::: "memory");        // done with the others' shared memory
    // how many of the tokens equal to tau the prefix takes (at least one: mass{w > tau} < target)
    unsigned long long n_ties = 1ull;
    int all_ties = 0;
#pragma unroll
    for (int r = 0; r < kRowMaxCluster; ++r) all_ties += n_of[r];
    if (all_ties > 1) {
        const unsigned long long tau_fx = fixed_point(tau, 44);
        n_ties = max(1ull, tau_fx ? (target_fx - mass_above + tau_fx - 1ull) / tau_fx : ~0ull);
    }
    // every CTA forms the same masses of all CTAs' members: above tau, and the ties that are in
    double Z = 0.0;
    unsigned long long tie_total = 0ull, tie_base = 0ull;
#pragma unroll
    for (int r = 0; r < kRowMaxCluster; ++r) {
        const unsigned long long k = (unsigned long long)n_of[r], room = n_ties > tie_total ? n_ties - tie_total : 0ull;
        if (r == rank) tie_base = tie_total;
        mass_of[r] += (double)(k < room ? k : room) * (double)tau;
        tie_total += k;
        Z += mass_of[r];
    }
    // Where order matters, every thread owns a contiguous run of the slice (an odd number of entries, so that the 32
    // runs of a warp start in different banks): vocabulary order over CTAs and threads.
    const int per = ((slice + kRowThreads - 1) / kRowThreads) | 1;
    const int e0 = min(n, t * per), e1 = min(n, e0 + per);
    if (tie_total > n_ties) {
        // ties past the prefix are no members: their weight goes to zero where it stands
        __syncthreads();                       // the last reads of s_warp_ties
        int ties = 0;
        for (int i = e0; i < e1; ++i) ties += s_w[i] == tau ? 1 : 0;
        int incl = ties;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) s_warp_ties[warp] = incl;
        __syncthreads();
        unsigned long long k = tie_base + (unsigned long long)(incl - ties);
        for (int w = 0; w < warp; ++w) k += (unsigned long long)s_warp_ties[w];
        if (ties > 0)
            for (int i = e0; i < e1; ++i)
                if (s_w[i] == tau && k++ >= n_ties) s_w[i] = 0.f;
    }
    // ---- the draw: the first CTA, thread and entry whose running mass exceeds the target (the last one with mass
    // where rounding pushes the target past the end)
    const double target = (double)p.u[row] * Z;
    double base = 0.0, run_cta = 0.0;
    int pick = -1, pick_last = 0;
#pragma unroll
    for (int r = 0; r < kRowMaxCluster; ++r) {
        if (mass_of[r] > 0.0) {
            pick_last = r;
            if (pick < 0 && run_cta + mass_of[r] > target) { pick = r; base = run_cta; }
        }
        run_cta += mass_of[r];
    }
    const bool past_end = pick < 0;
    if (past_end) pick = pick_last;
    if (pick == rank) {
        double mine = 0.0;
        for (int i = e0; i < e1; ++i) { const float w = s_w[i]; if (w >= tau) mine += (double)w; }
        double incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        __syncthreads();                       // the last reads of s_warp_mass
        if (lane == 31) s_warp_mass[warp] = incl;
        __syncthreads();
        double warp_base = base;
#pragma unroll
        for (int w = 0; w < kRowWarps; ++w) if (w < warp) warp_base += s_warp_mass[w];
        if (mine > 0.0) {
            atomicMax(&s_owner_last, t);
            if (!past_end && warp_base + incl > target) atomicMin(&s_owner, t);
        }
        __syncthreads();
        const bool by_mass = s_owner != 0x7fffffff;
        if (t == (by_mass ? s_owner : s_owner_last)) {
            double run = warp_base + (incl - mine);
            int first = -1, last = -1;
            for (int i = e0; i < e1; ++i) {
                const float w = s_w[i];
                if (w >= tau) {
                    run += (double)w;
                    last = i;
                    if (by_mass && run > target) { first = i; break; }
                }
            }
            p.tokens[row] = v0 + (first >= 0 ? first : last);
        }
    }
    if (p.probs_out) {
        __syncthreads();                       // weights set to zero above
        const float inv_Z = (float)(1.0 / Z);
        float* out = p.probs_out + (size_t)row * p.V + v0;
        auto prob = [&](float w) { return w >= tau ? w * inv_Z : 0.f; };
        if ((reinterpret_cast<uintptr_t>(out) & 15u) == 0 && n % 4 == 0) {
            for (int i = t; i < n4; i += kRowThreads) {
                const float4 y = reinterpret_cast<const float4*>(s_w)[i];
                __stcs(reinterpret_cast<float4*>(out) + i, make_float4(prob(y.x), prob(y.y), prob(y.z), prob(y.w)));
            }
        } else {
            for (int i = t; i < n; i += kRowThreads) __stcs(out + i, prob(s_w[i]));
        }
    }
    if (n_ctas > 1) asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

}  // namespace

// CTAs per row: as few as hold the row two to an SM (one to an SM for the longest rows), then more while rows are so
// few that SMs would stay idle and a CTA keeps at least 2,048 entries (below that the cluster's barriers cost more than
// the shorter walks bring).
static int row_cluster(int rows, int V) {
    int c = 1;
    while (c < kRowMaxCluster && V > c * kRowPairSlice) c *= 2;
    while (c < kRowMaxCluster && (long)rows * c * 2 <= device_sm_count() && V >= 2 * c * 2048) c *= 2;
    return c;
}

cudaError_t launch_top_p(const TopPParams& p, cudaStream_t stream) {
    cudaError_t e;
    if (p.V <= kRowMaxSlice * kRowMaxCluster) {
        const int c = row_cluster(p.rows, p.V);
        const int slice = ((p.V + c - 1) / c + 3) / 4 * 4;
        const size_t smem = (size_t)slice * sizeof(float);
        e = cudaFuncSetAttribute(top_p_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kRowMaxSlice * sizeof(float)));
        if (e != cudaSuccess) return e;
        const dim3 grid((unsigned)((long)p.rows * c));
        e = c == 1 ? launch_pdl(top_p_cluster_kernel, grid, dim3(kRowThreads), smem, stream, p, c, slice)
                   : launch_pdl_cluster(top_p_cluster_kernel, grid, dim3(kRowThreads), smem, stream, c, p, c, slice);
    } else {
        e = launch_pdl(top_p_kernel, dim3(p.rows), dim3(kTopPThreads), 0, stream, p);
    }
    if (e != cudaSuccess) return e;
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace massv
