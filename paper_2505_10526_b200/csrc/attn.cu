// Verify attention: the gamma+1 block rows of every sequence attend the paged
// KV cache (Sec. 2.1: the target scores positions t+1..t+gamma+1 in one forward
// call; Sec. 2.2: the cache holds image tokens, then text, then the block).
//
// The scan over the cache is bound by HBM.  All G*(gamma+1) query rows that share
// a KV head are processed by the same CTA so that every K/V byte is read once.
// Two schedules (see launch_verify_attn): work items = (sequence, KV head, chunk of
// kv_chunk positions) on a grid (max_chunks, Hkv, B), where CTAs whose chunk lies beyond
// the sequence retire at once; or, at head_dim 256, a persistent grid that cuts the line of
// all tiles into equal ranges (attn_flat_kernel).  Inside a CTA a
// producer warp streams 64-token (32-token at d = 256) K/V tiles page by page with TMA (16 x 64 boxes,
// 128-byte swizzle) into an mbarrier ring; consumer warps run
// Q K^T and P V on warp-level tensor-core MMAs (m16n8k16, bf16 -> fp32) with an
// online softmax in registers: warp (mt, ts) owns 16 query rows and a 64/TS-token
// slice of every tile.  Partial (max, sum, O) of the warps are merged through
// shared memory; sequences that span several chunks are merged by a second
// kernel.  The block's own K/V rows are appended by the CTA whose chunk holds
// their positions.  All reductions have a fixed order.
#include "kernels.cuh"
#include "ptx.cuh"

namespace massv {

namespace {

constexpr int kChunkAlign = 64;      // kv_chunk granularity (a multiple of every tile size)
constexpr int kMaxChunkPages = 256;  // kv_chunk <= 4096 tokens
constexpr float kRefDrop = 6.f;      // binary orders that a slice's reference may lie below the running maximum

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
// d += a(16x16, row) * b(16x8, col), bf16 inputs, fp32 accumulate
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&v);
}


// Byte offset of the 16-byte unit `unit` (0..7) of row `row` inside a region of
// 128-byte rows laid out with the 128-byte swizzle (what TMA writes).
__device__ __forceinline__ uint32_t swz(int row, int unit) { return (uint32_t)(row * 128 + ((unit ^ (row & 7)) << 4)); }

// TILE = tokens per pipeline stage (32 or 64).  DEEP: the CTA has an SM to itself (five
// warps), so the ring is twice as deep to keep enough bytes in flight.
template <int D, int TILE, bool DEEP>
struct AttnCfg {
    static constexpr int kChunks = D / 64;                 // 64-element column groups of a row
    static constexpr int kRegion = TILE * 128;             // bytes of one (TILE tokens x 64 elements) region
    static constexpr int kBytesK = kChunks * kRegion;
    static constexpr int kStageBytes = 2 * kBytesK;        // K then V
    static constexpr int kStages = DEEP ? 6 : ((D == 64) ? 4 : 3);
};

// One tile of K/V for a warp: its 16 query rows (group mt) against its TILE/TS tokens (slice ts) of the tile at `kst` (K, then
// V), the online softmax carried in (o, m_run, l_run, r_run): l_run is relative to the running maximum m_run, o to r_run, the
// maximum of the latest slice (kept within kRefDrop binary orders of m_run, so that o cannot outgrow its range).  The
// largest weight of every slice is then exactly 1, and it is the heaviest weights whose rounding to bf16 shows in the
// output.  With the running maximum as the reference only the maxima of a prefix were exact, so the error of a row depended
// on the number of cuts its context had (32 x 8 pairs of 2k - 8k positions, error against 64 bits relative to the norm: 1.43e-3
// with the fixed chunks, 1.47e-3 with the longer runs of the balanced schedule, 1.02e-3 with either now).  page_of(position) is the page that holds it (asked for the block's
// own positions only: they are appended here).
template <int D, int MT, int TS, int TILE, typename PageOf>
__device__ __forceinline__ void attend_tile(const AttnParams& p, int b, int g, int L, int c_end, int tile_start, uint8_t* kst, uint32_t q_base,
                                            const uint32_t (&qf)[D <= 128 ? D / 16 : 1][4], int mt, int ts, int lane, int j0, int j1, float scale_log2,
                                            PageOf&& page_of, float (&o)[D / 8][4], float (&m_run)[2], float (&l_run)[2], float (&r_run)[2]) {
    constexpr int kTile = TILE, NT = TILE / TS, RP = MT * 16;
    constexpr int kRegion = TILE * 128, kBytesK = (D / 64) * kRegion;
    constexpr bool kQInRegs = D <= 128;
    const int n_ctx = L + p.R;
    const int lm = lane >> 3, lr = lane & 7;      // ldmatrix lane roles: matrix (lane >> 3), row (lane & 7) inside it
    const int valid = min(kTile, c_end - tile_start);
    uint8_t* vst = kst + kBytesK;
    if (tile_start + kTile > L) {
        constexpr int UPR = D / 8;
        // Append: the block's K/V rows (positions L .. L+gamma) are not in the cache yet.
        // The warp that owns those tokens puts them into the tile in shared memory, and
        // the mt == 0 warp also stores them to their page slots.
        const int p_first = max(L, tile_start + ts * NT), p_last = min(n_ctx, tile_start + ts * NT + NT);
        // (All rows in flight at once: one after the other through registers, a pair of six rows took six memory latencies.)
        for (int i = lane; i < (p_last - p_first) * UPR; i += 32) {
            const int pos = p_first + i / UPR, u = i % UPR, row = pos - tile_start;
            const size_t src = (((size_t)b * p.R + (pos - L)) * p.Hkv + g) * D + u * 8;
            cp_async_16(kst + (u / 8) * kRegion + swz(row, u % 8), p.k_new + src);
            cp_async_16(vst + (u / 8) * kRegion + swz(row, u % 8), p.v_new + src);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        if (mt == 0) {
            for (int i = lane; i < (p_last - p_first) * UPR; i += 32) {          // the units this lane has copied
                const int pos = p_first + i / UPR, u = i % UPR, row = pos - tile_start;
                const int pid = page_of(pos);
                if (pid >= 0 && pid < p.num_pages) {
                    const size_t dst = (((size_t)pid * p.Hkv + g) * kPageSize + (pos % kPageSize)) * D + u * 8;
                    *reinterpret_cast<uint4*>(p.k_pages + dst) = *reinterpret_cast<const uint4*>(kst + (u / 8) * kRegion + swz(row, u % 8));
                    *reinterpret_cast<uint4*>(p.v_pages + dst) = *reinterpret_cast<const uint4*>(vst + (u / 8) * kRegion + swz(row, u % 8));
                }
            }
        }
        // Rows past the end of the context hold stale bytes; their weights are zero, but
        // 0 * NaN would still poison P V, so clear the V rows this warp will read.
        const int first = max(valid, ts * NT), last = ts * NT + NT;
        for (int i = lane; i < (last - first) * UPR; i += 32) {
            const int row = first + i / UPR, u = i % UPR;
            *reinterpret_cast<uint4*>(vst + (u / 8) * kRegion + swz(row, u % 8)) = make_uint4(0u, 0u, 0u, 0u);
        }
        // The balanced schedule refills this stage for its next pair: these stores have to be ordered ahead of the TMA's
        // (async-proxy) writes to the same bytes, which the mbarrier between the two does not do.
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
    }
    const uint32_t k_base = smem_u32(kst), v_base = smem_u32(vst);

    // ---- S = Q K^T for this warp's 16 rows x NT tokens
    float sacc[NT / 8][4];
#pragma unroll
    for (int n = 0; n < NT / 8; ++n) { sacc[n][0] = sacc[n][1] = sacc[n][2] = sacc[n][3] = 0.f; }
#pragma unroll
    for (int kk = 0; kk < D / 16; ++kk) {
        uint32_t a[4];
        if (kQInRegs) {
            a[0] = qf[kk][0]; a[1] = qf[kk][1]; a[2] = qf[kk][2]; a[3] = qf[kk][3];
        } else {
            const int row = mt * 16 + (lm & 1) * 8 + lr, unit = (kk & 3) * 2 + (lm >> 1);
            ldmatrix_x4(a, q_base + (kk >> 2) * (RP * 128) + swz(row, unit));
        }
#pragma unroll
        for (int tg = 0; tg < NT / 16; ++tg) {
            uint32_t bf[4];
            const int tok = ts * NT + tg * 16 + (lm >> 1) * 8 + lr, unit = (kk & 3) * 2 + (lm & 1);
            ldmatrix_x4(bf, k_base + (kk >> 2) * kRegion + swz(tok, unit));
            mma_bf16(sacc[2 * tg], a, bf[0], bf[1]);
            mma_bf16(sacc[2 * tg + 1], a, bf[2], bf[3]);
        }
    }

    // ---- scale, causal mask, online softmax
    // some position in the tile is hidden from some block row: ahead of row 0, or (with a
    // window) older than the last row's lower bound
    const bool need_mask = tile_start + kTile > L + 1 || (p.window > 0 && tile_start < n_ctx - p.window);
    float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
    for (int n = 0; n < NT / 8; ++n) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            float sv = sacc[n][e] * scale_log2;
            if (need_mask) {
                const int pos = tile_start + ts * NT + n * 8 + 2 * (lane & 3) + (e & 1);
                const int row_pos = L + (e < 2 ? j0 : j1);
                if (pos > row_pos || (p.window > 0 && pos < row_pos - p.window + 1)) sv = -INFINITY;
            }
            sacc[n][e] = sv;
            if (e < 2) mx0 = fmaxf(mx0, sv); else mx1 = fmaxf(mx1, sv);
        }
    }
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
    mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
    mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
    const float mn0 = fmaxf(m_run[0], mx0), mn1 = fmaxf(m_run[1], mx1);
    const float rn0 = fmaxf(mx0, mn0 - kRefDrop), rn1 = fmaxf(mx1, mn1 - kRefDrop);
    const float ms0 = rn0 == -INFINITY ? 0.f : rn0, ms1 = rn1 == -INFINITY ? 0.f : rn1;
    const float corr0 = ex2_ftz(r_run[0] - ms0), corr1 = ex2_ftz(r_run[1] - ms1);
    r_run[0] = rn0; r_run[1] = rn1;
    float ls0 = 0.f, ls1 = 0.f;
    uint32_t pa[NT / 16][4];
#pragma unroll
    for (int n = 0; n < NT / 8; ++n) {
        const float p0 = exp2f(sacc[n][0] - ms0), p1 = exp2f(sacc[n][1] - ms0);
        const float p2 = exp2f(sacc[n][2] - ms1), p3 = exp2f(sacc[n][3] - ms1);
        ls0 += p0 + p1; ls1 += p2 + p3;
        // accumulator layout -> A-operand layout of the P V product
        pa[n >> 1][(n & 1) * 2 + 0] = pack_bf16(p0, p1);
        pa[n >> 1][(n & 1) * 2 + 1] = pack_bf16(p2, p3);
    }
    const float mt0 = mn0 == -INFINITY ? 0.f : mn0, mt1 = mn1 == -INFINITY ? 0.f : mn1;
    if (__any_sync(0xffffffffu, mn0 > m_run[0] || mn1 > m_run[1])) {
        l_run[0] *= ex2_ftz(m_run[0] - mt0); l_run[1] *= ex2_ftz(m_run[1] - mt1);
        m_run[0] = mn0; m_run[1] = mn1;
    }
    l_run[0] += ls0 * ex2_ftz(rn0 - mt0);
    l_run[1] += ls1 * ex2_ftz(rn1 - mt1);
#pragma unroll
    for (int n = 0; n < D / 8; ++n) { o[n][0] *= corr0; o[n][1] *= corr0; o[n][2] *= corr1; o[n][3] *= corr1; }

    // ---- O += P V
#pragma unroll
    for (int tk = 0; tk < NT / 16; ++tk) {
#pragma unroll
        for (int dp = 0; dp < D / 16; ++dp) {
            uint32_t bf[4];
            const int tok = ts * NT + tk * 16 + (lm & 1) * 8 + lr, du = dp * 2 + (lm >> 1);
            ldmatrix_x4_trans(bf, v_base + (du >> 3) * kRegion + swz(tok, du & 7));
            mma_bf16(o[2 * dp], pa[tk], bf[0], bf[1]);
            mma_bf16(o[2 * dp + 1], pa[tk], bf[2], bf[3]);
        }
    }
}

// The accumulator relative to the running maximum, as the merges take it.
template <int D>
__device__ __forceinline__ void settle(float (&o)[D / 8][4], const float (&m_run)[2], const float (&r_run)[2]) {
    const float f0 = m_run[0] == -INFINITY ? 0.f : exp2f(r_run[0] - m_run[0]), f1 = m_run[1] == -INFINITY ? 0.f : exp2f(r_run[1] - m_run[1]);
#pragma unroll
    for (int n = 0; n < D / 8; ++n) { o[n][0] *= f0; o[n][1] *= f0; o[n][2] *= f1; o[n][3] *= f1; }
}

// Two CTAs should share an SM (one CTA's set-up and merge hide behind the other's
// streaming).  Each scheduler owns a quarter of the register file and a CTA's warps are
// dealt round-robin, so that needs at most four warps per CTA, producer included.
template <int D, int MT, int TS, int TILE>
__global__ void __launch_bounds__((MT * TS + 1) * 32, (MT * TS + 1) <= 4 ? 2 : 1)
attn_split_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const AttnParams p) {
    using Cfg = AttnCfg<D, TILE, (MT * TS + 1 > 4)>;
    constexpr int kTile = TILE;
    constexpr int NW = MT * TS;            // consumer warps
    constexpr int RP = MT * 16;            // padded query rows
    constexpr int NCH = Cfg::kChunks;
    constexpr bool kQInRegs = D <= 128;

    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[Cfg::kStages];
    __shared__ __align__(8) uint64_t empty_bar[Cfg::kStages];
    __shared__ int s_pages[kMaxChunkPages];
    __shared__ int abort_flag;

    const int chunk = blockIdx.x, g = blockIdx.y, b = blockIdx.z;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();
    const int L = p.seq_lens[b];
    if (L < 0 || L + p.R > p.max_pages * kPageSize) {            // no room for the block: skip the sequence
        if (chunk == 0 && g == 0 && threadIdx.x == 0) set_status(p.dev_status, MASSV_ERR_CAPACITY);
        return;
    }
    const int n_ctx = L + p.R;
    if (chunk * p.kv_chunk >= n_ctx) return;
    // Sliding window: block row j (position L + j) sees positions L + j - window + 1 .. L + j, so
    // nothing before row 0's lower bound is needed.  Chunks wholly before it retire, and the
    // first needed chunk starts at the tile that holds the bound.
    const int lo_min = p.window > 0 ? max(0, L - p.window + 1) : 0;
    const int first_chunk = lo_min / p.kv_chunk;
    if (chunk < first_chunk) return;
    int c_begin = chunk * p.kv_chunk;
    if (chunk == first_chunk) c_begin += ((lo_min - c_begin) / kTile) * kTile;
    const int c_end = min(n_ctx, chunk * p.kv_chunk + p.kv_chunk);
    const int n_tiles = (c_end - c_begin + kTile - 1) / kTile;
    const int n_chunks_b = (n_ctx + p.kv_chunk - 1) / p.kv_chunk - first_chunk;     // chunks that take part
    const int G = p.Hq / p.Hkv;
    const int rows = G * p.R;

    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* q_smem = smem + Cfg::kStages * Cfg::kStageBytes;    // [NCH][RP rows][128 B], swizzled

    if (threadIdx.x == 0) {
        for (int s = 0; s < Cfg::kStages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], NW); }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    {   // page ids of this chunk and the query rows (row r = block_row * G + head_in_group)
        const int n_pages = (c_end - c_begin + kPageSize - 1) / kPageSize;
        for (int i = threadIdx.x; i < n_pages; i += blockDim.x)
            s_pages[i] = p.page_table[(size_t)b * p.max_pages + c_begin / kPageSize + i];
        constexpr int UPR = D / 8;   // 16-byte units per row
        for (int i = threadIdx.x; i < RP * UPR; i += blockDim.x) {
            const int r = i / UPR, u = i % UPR;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (r < rows) {
                const int j = r / G, hh = r % G;
                v = *reinterpret_cast<const uint4*>(p.q + (((size_t)b * p.R + j) * p.Hq + g * G + hh) * D + u * 8);
            }
            *reinterpret_cast<uint4*>(q_smem + (u / 8) * (RP * 128) + swz(r, u % 8)) = v;
        }
    }
    __syncthreads();
    volatile int* abort_ptr = &abort_flag;

    float o[D / 8][4];
    float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f}, r_run[2] = {-INFINITY, -INFINITY};
    const int mt = warp / TS, ts = warp % TS;

    if (warp == NW) {
        // ------------------------------------------------ TMA producer
        // A tile is 2 * (d/64) boxes per page.  One box per lane: a single thread issuing them one
        // after the other cannot keep an SM's share of HBM busy when the CTA has the SM to itself.
        uint64_t policy;
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
        for (int t = 0; t < n_tiles; ++t) {
            const int s = t % Cfg::kStages;
            const uint32_t ph = ((uint32_t)(t / Cfg::kStages)) & 1u;
            int freed = 0;
            if (lane == 0) freed = mbar_wait(&empty_bar[s], ph ^ 1u, abort_ptr) ? 1 : 0;
            freed = __shfl_sync(0xffffffffu, freed, 0);
            if (!freed) break;
            const int tile_start = c_begin + t * kTile;
            int n_pg = (c_end - tile_start + kPageSize - 1) / kPageSize;
            if (n_pg > kTile / kPageSize) n_pg = kTile / kPageSize;
            uint8_t* kdst = smem + (size_t)s * Cfg::kStageBytes;
            if (lane == 0) mbar_expect_tx(&full_bar[s], (uint32_t)(n_pg * NCH * 2048 * 2));
            __syncwarp();
            for (int i = lane; i < n_pg * NCH * 2; i += 32) {
                const int is_v = i & 1, dc = (i >> 1) % NCH, pg = i / (2 * NCH);
                int pid = s_pages[t * (kTile / kPageSize) + pg];
                if (pid < 0 || pid >= p.num_pages) { set_status(p.dev_status, MASSV_ERR_CAPACITY); pid = 0; }
                const int row = (pid * p.Hkv + g) * kPageSize;
                tma_load_2d(kdst + is_v * Cfg::kBytesK + dc * Cfg::kRegion + pg * 2048, is_v ? &map_v : &map_k, dc * 64, row,
                            &full_bar[s], policy);
            }
        }
        if (lane == 0 && *abort_ptr) {
            for (int i = 0; i < 64; ++i) __nanosleep(2000);   // let copies in flight land
        }
    } else {
        // ------------------------------------------------ consumers
#pragma unroll
        for (int n = 0; n < D / 8; ++n) { o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f; }
        const float scale_log2 = p.scale * 1.4426950408889634f;
        const int r0 = mt * 16 + (lane >> 2), r1 = r0 + 8;
        // block row of each of this thread's two query rows (padding rows behave like the last block row)
        const int j0 = r0 < rows ? r0 / G : p.R - 1, j1 = r1 < rows ? r1 / G : p.R - 1;
        const uint32_t q_base = smem_u32(q_smem);
        // ldmatrix lane roles: matrix (lane >> 3), row (lane & 7) inside it
        const int lm = lane >> 3, lr = lane & 7;
        uint32_t qf[kQInRegs ? D / 16 : 1][4];
        if (kQInRegs) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
                const int row = mt * 16 + (lm & 1) * 8 + lr, unit = (kk & 3) * 2 + (lm >> 1);
                ldmatrix_x4(qf[kk], q_base + (kk >> 2) * (RP * 128) + swz(row, unit));
            }
        }
        bool ok = true;
        for (int t = 0; t < n_tiles && ok; ++t) {
            const int s = t % Cfg::kStages;
            const uint32_t ph = ((uint32_t)(t / Cfg::kStages)) & 1u;
            if (!mbar_wait(&full_bar[s], ph, abort_ptr)) { ok = false; break; }
            const int tile_start = c_begin + t * kTile;
            attend_tile<D, MT, TS, TILE>(p, b, g, L, c_end, tile_start, smem + (size_t)s * Cfg::kStageBytes, q_base, qf, mt, ts, lane, j0, j1, scale_log2,
                                         [&](int pos) { return s_pages[(pos - c_begin) / kPageSize]; }, o, m_run, l_run, r_run);
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty_bar[s]);
        }
        settle<D>(o, m_run, r_run);
        l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 1);
        l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 2);
        l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 1);
        l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 2);
    }

    // ---------------------------------------------------- merge the warps' partial results
    __syncthreads();                         // every tile has been consumed: the ring can be reused
    pdl_trigger();
    float* st_o = reinterpret_cast<float*>(smem);            // [TS][RP][D]
    float* st_m = st_o + TS * RP * D;                        // [TS][RP]
    float* st_l = st_m + TS * RP;
    if (warp < NW) {
        const int r0 = mt * 16 + (lane >> 2), r1 = r0 + 8;
        float* base = st_o + (size_t)ts * RP * D;
#pragma unroll
        for (int n = 0; n < D / 8; ++n) {
            const int c = n * 8 + 2 * (lane & 3);
            *reinterpret_cast<float2*>(base + r0 * D + c) = make_float2(o[n][0], o[n][1]);
            *reinterpret_cast<float2*>(base + r1 * D + c) = make_float2(o[n][2], o[n][3]);
        }
        if ((lane & 3) == 0) {
            st_m[ts * RP + r0] = m_run[0]; st_l[ts * RP + r0] = l_run[0];
            st_m[ts * RP + r1] = m_run[1]; st_l[ts * RP + r1] = l_run[1];
        }
    }
    __syncthreads();
    if (abort_flag) {
        if (threadIdx.x == 0) set_status(p.dev_status, MASSV_ERR_TIMEOUT);
        return;
    }
    const bool single = n_chunks_b == 1;
    const size_t item = ((size_t)b * p.Hkv + g) * p.max_chunks + chunk;
    for (int i = threadIdx.x; i < rows * (D / 4); i += blockDim.x) {
        const int r = i / (D / 4), c = (i % (D / 4)) * 4;
        float M = -INFINITY;
#pragma unroll
        for (int w = 0; w < TS; ++w) M = fmaxf(M, st_m[w * RP + r]);
        float Lsum = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < TS; ++w) {
            const float mw = st_m[w * RP + r];
            const float f = mw == -INFINITY ? 0.f : exp2f(mw - M);
            Lsum += st_l[w * RP + r] * f;
            const float4 v = *reinterpret_cast<const float4*>(st_o + ((size_t)w * RP + r) * D + c);
            acc.x += v.x * f; acc.y += v.y * f; acc.z += v.z * f; acc.w += v.w * f;
        }
        if (single) {
            const int j = r / G, hh = r % G;
            const size_t dst = (((size_t)b * p.R + j) * p.Hq + g * G + hh) * D + c;
            const float inv = 1.f / Lsum;
            acc.x *= inv; acc.y *= inv; acc.z *= inv; acc.w *= inv;
            uint2 packed;
            packed.x = pack_bf16(acc.x, acc.y);
            packed.y = pack_bf16(acc.z, acc.w);
            *reinterpret_cast<uint2*>(p.out + dst) = packed;
            if (p.out_f32) *reinterpret_cast<float4*>(p.out_f32 + dst) = acc;
            if (p.lse && c == 0) p.lse[((size_t)b * p.R + j) * p.Hq + g * G + hh] = (M + log2f(Lsum)) * 0.6931471805599453f;
        } else {
            *reinterpret_cast<float4*>(p.part_o + (item * RP + r) * D + c) = acc;
            if (c == 0) { p.part_ml[(item * RP + r) * 2] = M; p.part_ml[(item * RP + r) * 2 + 1] = Lsum; }
        }
    }
}

// ---- The balanced schedule (as in attn_umma.cu): the tiles of all (sequence, KV head) pairs form one line ordered by
// (sequence, head, position), a persistent grid cuts it into equal ranges, and a CTA leaves at most two pieces of cut pairs to
// attn_flat_combine_kernel, in the layout the accumulators have in registers.  The ring runs on across the pairs of a
// range: while the compute warps merge and write one pair, the producer is already filling the next one's tiles.
// Against a grid of fixed chunks every CTA streams the same bytes whatever the mix of lengths and window bounds, and pays
// its set-up once.
// The line is measured in tiles, and a pair's set-up and merge count as kPairUnits tiles ahead of its own: a sequence of a few
// positions is one tile for each of its heads, and a CTA that got a dozen such pairs for a dozen tiles of one long pair held
// all others up.  64 x 8 pairs of 1 - 512 positions: 81 us with 0 units, 58, 51, 50 and 50 with 2, 4, 6 and 8; 32 x 8 of
// 2k - 8k: 225, 225, 223, 223, 231; the same with a window of 1,024: 61.3, 62.1, 62.0, 63.3, 63.7.
constexpr int kPairUnits = 4;
constexpr int kPairSlack = 6;              // (see flat_range)
// By one warp: range[0], range[1] = this CTA's units of the line, range[2] = units per CTA.  Equal ranges; but a pair per CTA
// (range[2] = kFlatWholePairs) where the longest pair is at most kPairSlack units (fewer for short ranges) longer than a range - the window of a local
// layer, contexts of one length - so that nothing is cut, written as pieces and merged.  Call times, equal ranges -> a pair per CTA: 256 pairs
// of 12 rows, window 1,024 (5 units) 57 -> 53 us, window 512 38 -> 33, 1,000 positions 57 -> 46; 128 pairs of 24 rows, window 1,024 49 -> 45,
// 4,000 positions (17 units) 127 -> 134.  (The tcgen05 kernel keeps its ranges: the longer its runs, the further its running reference leaves
// the weights of later tiles from exact ones.)
__device__ __forceinline__ void flat_range(const int* cum, int batch, int kv_heads, int longest, int* range) {
    __syncwarp();
    if ((threadIdx.x & 31) != 0) return;
    const int total = cum[batch] * kv_heads, ctas = (int)gridDim.x, at = (int)blockIdx.x;
    int per = max(1, (total + ctas - 1) / ctas);
    int first = min(total, at * per), end = min(total, first + per);
    if (batch * kv_heads <= ctas && longest <= per + min(kPairSlack, 1 + per / kPairSlack)) {
        const int b = at / kv_heads, g = at % kv_heads, n = b < batch ? cum[b + 1] - cum[b] : 0;
        first = b < batch ? cum[b] * kv_heads + g * n : total;
        end = first + n;
        per = kFlatWholePairs;
    }
    range[0] = first; range[1] = end; range[2] = per;
}
template <int D, int MT, int TILE>
struct FlatCfg {
    static constexpr int kTS = 2;                          // warps that share 16 query rows, each with half of a tile's tokens
    static constexpr int kWarps = MT * kTS;
    static constexpr int kChunks = D / 64;
    static constexpr int kRegion = TILE * 128;
    static constexpr int kBytesK = kChunks * kRegion;
    static constexpr int kStageBytes = 2 * kBytesK;
    // up to 16 rows: two CTAs per SM with three stages each; above, one CTA needs the shared memory and the warps alone
    static constexpr int kStages = MT == 1 ? 3 : (MT == 4 ? 5 : 6);
    static constexpr int kCtasPerSm = MT == 1 ? 2 : 1;
    static constexpr int kQBytes = MT * 16 * D * 2;
    static constexpr int kSmem = kStages * kStageBytes + kQBytes + 1024;      // and (B + 1) ints
};

// WHOLE: a pair per CTA is possible, and flat_range decides.  (A kernel of its own: the decision costs a short call 0.2 us, 4 x 8 pairs of
// 41 - 65 positions 11.20 -> 11.40.)
template <int D, int MT, int TILE, bool WHOLE>
__global__ void __launch_bounds__((FlatCfg<D, MT, TILE>::kWarps + 1) * 32, FlatCfg<D, MT, TILE>::kCtasPerSm)
attn_flat_kernel(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_q,
                 const AttnParams p) {
    using Cfg = FlatCfg<D, MT, TILE>;
    static_assert(D == 256, "the exchange between the two warps of a row group goes through the query rows' space");
    constexpr int NW = Cfg::kWarps, RP = MT * 16, TS = Cfg::kTS, E = Cfg::kStages, NCH = Cfg::kChunks, UPR = D / 8;
    constexpr int PPT = TILE / kPageSize, GROUP = 32 / PPT;           // pages per tile; tiles whose page ids fit one register per lane
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t full_bar[E], empty_bar[E];
    __shared__ float s_m[NW][16], s_l[NW][16];
    __shared__ int abort_flag, s_range[3];

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int G = p.Hq / p.Hkv, rows = G * p.R;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* q_smem = smem + E * Cfg::kStageBytes;                   // [NCH][RP rows][128 B], swizzled
    int* s_cum = reinterpret_cast<int*>(q_smem + Cfg::kQBytes);      // tiles of sequences 0 .. b-1 (per KV head)
    if (threadIdx.x == 0) {
        for (int s = 0; s < E; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], NW); }
        abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    pdl_wait();

    // units per pair of every sequence, then an exclusive prefix sum over the batch
    auto first_tile = [&](int L) { return (p.window > 0 ? max(0, L - p.window + 1) : 0) / TILE; };
    for (int i = threadIdx.x; i < p.B; i += blockDim.x) {
        const int L = p.seq_lens[i];
        int n = 0;
        if (L < 0 || L + p.R > p.max_pages * kPageSize) {            // no room for the block: skip the sequence
            if (blockIdx.x == 0) set_status(p.dev_status, MASSV_ERR_CAPACITY);
        } else {
            n = (L + p.R + TILE - 1) / TILE - first_tile(L) + kPairUnits;
        }
        s_cum[i + 1] = n;
    }
    if (threadIdx.x == 0) s_cum[0] = 0;
    __syncthreads();
    if (warp == 0) {
        const int per = (p.B + 31) / 32;
        const int i0 = min(p.B, lane * per), i1 = min(p.B, i0 + per);
        int local = 0, longest = 0;
        for (int i = i0; i < i1; ++i) { local += s_cum[i + 1]; longest = max(longest, s_cum[i + 1]); }
        int incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        int run = incl - local;
        for (int i = i0; i < i1; ++i) { run += s_cum[i + 1]; s_cum[i + 1] = run; }
        if constexpr (WHOLE) flat_range(s_cum, p.B, p.Hkv, __reduce_max_sync(0xffffffffu, longest), s_range);
    }
    __syncthreads();
    const int total = s_cum[p.B] * p.Hkv;
    const int per_cta = WHOLE ? s_range[2] : max(1, (total + (int)gridDim.x - 1) / (int)gridDim.x);
    if (blockIdx.x == 0) {          // what the merge kernel needs to find the pieces of a pair
        for (int i = threadIdx.x; i <= p.B; i += blockDim.x) p.flat_meta[2 + i] = s_cum[i];
        if (threadIdx.x == 0) { p.flat_meta[0] = per_cta; p.flat_meta[1] = kPairUnits; }
    }
    const int f_first = WHOLE ? s_range[0] : min(total, (int)blockIdx.x * per_cta), f_end = WHOLE ? s_range[1] : min(total, f_first + per_cta);
    volatile int* abort_ptr = &abort_flag;

    // Piece of work at unit f of the line: a run of tiles of one pair, up to this CTA's end (none where that lies ahead of them).
    struct Piece { int b, g, L, c_begin, c_end, n_tiles, n_units; bool whole; };
    int b_hint = 0;
    auto piece_at = [&](int f) {
        int lo = b_hint, hi = p.B - 1;                               // largest b with Hkv * cum[b] <= f
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (s_cum[mid] * p.Hkv <= f) lo = mid; else hi = mid - 1;
        }
        b_hint = lo;
        const int n_b = s_cum[lo + 1] - s_cum[lo], off = f - s_cum[lo] * p.Hkv;
        const int u0 = off % n_b, u1 = min(n_b, u0 + (f_end - f)), t0 = max(0, u0 - kPairUnits), t1 = max(0, u1 - kPairUnits);
        Piece w;
        w.b = lo; w.g = off / n_b; w.L = p.seq_lens[lo];
        const int tile_lo = first_tile(w.L);
        w.c_begin = (tile_lo + t0) * TILE;
        w.c_end = min(w.L + p.R, (tile_lo + t1) * TILE);
        w.n_tiles = t1 - t0;
        w.n_units = u1 - u0;
        w.whole = t0 == 0 && u1 == n_b;
        return w;
    };

    if (warp == NW) {
        // ------------------------------------------------ TMA producer: one box per lane (16 per full tile)
        uint64_t policy;
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int f = f_first; f < f_end && ok;) {
            const Piece w = piece_at(f);
            f += w.n_units;
            if (w.n_tiles == 0) continue;
            // page ids travel in registers, lane l holding page 32 * group + l; the next group's are fetched a group ahead
            const int32_t* pt = p.page_table + (size_t)w.b * p.max_pages + w.c_begin / kPageSize;
            const int n_pages = (w.c_end - w.c_begin + kPageSize - 1) / kPageSize;
            int pid_cur = lane < n_pages ? pt[lane] : 0, pid_next = 32 + lane < n_pages ? pt[32 + lane] : 0;
            {
                // The pair's query rows travel through the ring ahead of its tiles (row r = block_row * G + head_in_group, and the
                // G heads of a block row are adjacent in memory: one box per block row and 64-element column group).
                int freed = 0;
                if (lane == 0) freed = mbar_wait(&empty_bar[s], ph ^ 1u, abort_ptr) ? 1 : 0;
                if (!__shfl_sync(0xffffffffu, freed, 0)) { ok = false; break; }
                if (lane == 0) mbar_expect_tx(&full_bar[s], (uint32_t)(rows * D * 2));
                __syncwarp();
                static_assert(kMaxRows * NCH <= 32, "one box per lane");
                const int j = lane / NCH, dc = lane % NCH;
                if (j < p.R)
                    tma_load_2d(smem + (size_t)s * Cfg::kStageBytes + dc * (RP * 128) + j * G * 128, &map_q, dc * 64, (w.b * p.R + j) * p.Hq + w.g * G,
                                &full_bar[s], policy);
                if (++s == E) { s = 0; ph ^= 1u; }
            }
            for (int t = 0; t < w.n_tiles; ++t) {
                if (t > 0 && t % GROUP == 0) {
                    pid_cur = pid_next;
                    const int nxt = (t / GROUP + 1) * 32 + lane;
                    pid_next = nxt < n_pages ? pt[nxt] : 0;
                }
                int freed = 0;
                if (lane == 0) freed = mbar_wait(&empty_bar[s], ph ^ 1u, abort_ptr) ? 1 : 0;
                if (!__shfl_sync(0xffffffffu, freed, 0)) { ok = false; break; }
                const int n_pg = min(PPT, n_pages - t * PPT);
                uint8_t* dst = smem + (size_t)s * Cfg::kStageBytes;
                if (lane == 0) mbar_expect_tx(&full_bar[s], (uint32_t)(n_pg * NCH * 2048 * 2));
                __syncwarp();
                const int is_v = lane & 1, dc = (lane >> 1) % NCH, pg = lane / (2 * NCH);
                static_assert(2 * NCH * PPT <= 32, "one box per lane");
                int pid = __shfl_sync(0xffffffffu, pid_cur, (t % GROUP) * PPT + min(pg, PPT - 1));
                if (pg < n_pg) {
                    if (pid < 0 || pid >= p.num_pages) { set_status(p.dev_status, MASSV_ERR_CAPACITY); pid = 0; }
                    tma_load_2d(dst + is_v * Cfg::kBytesK + dc * Cfg::kRegion + pg * 2048, is_v ? &map_v : &map_k, dc * 64,
                                (pid * p.Hkv + w.g) * kPageSize, &full_bar[s], policy);
                }
                if (++s == E) { s = 0; ph ^= 1u; }
            }
        }
        if (!ok && lane == 0) {
            for (int i = 0; i < 64; ++i) __nanosleep(2000);          // let copies in flight land
        }
    } else {
        // ------------------------------------------------ compute warps (one that gave up waiting still meets the barriers)
        auto sync_warps = [&]() { asm volatile("bar.sync 1, %0;" ::"n"(NW * 32) : "memory"); };
        const int mt = warp / TS, ts = warp % TS;
        const float scale_log2 = p.scale * 1.4426950408889634f;
        const int r0 = mt * 16 + (lane >> 2), r1 = r0 + 8;
        // block row of each of this thread's two query rows (padding rows behave like the last block row)
        const int j0 = r0 < rows ? r0 / G : p.R - 1, j1 = r1 < rows ? r1 / G : p.R - 1;
        const uint32_t q_base = smem_u32(q_smem);
        float4* exchange = reinterpret_cast<float4*>(q_smem + mt * 16 * D * 2) + lane;     // half of the columns of 16 rows
        const uint32_t no_q[1][4] = {{0u, 0u, 0u, 0u}};
        int s = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int f = f_first; f < f_end;) {
            const Piece w = piece_at(f);
            const size_t slot = (size_t)blockIdx.x * 2 + (f == f_first ? 0 : 1);
            f += w.n_units;
            if (w.n_tiles == 0) continue;
            // the pair's query rows, from their ring stage to their place (same layout; zeros past the last row)
            if (ok && !mbar_wait_warp(&full_bar[s], ph, abort_ptr)) ok = false;
            for (int i = threadIdx.x; i < RP * UPR; i += NW * 32) {
                const int r = (i / 8) % RP;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (r < rows) v = *reinterpret_cast<const uint4*>(smem + (size_t)s * Cfg::kStageBytes + (size_t)i * 16);
                *reinterpret_cast<uint4*>(q_smem + (size_t)i * 16) = v;
            }
            sync_warps();
            if (lane == 0) mbar_arrive(&empty_bar[s]);
            if (++s == E) { s = 0; ph ^= 1u; }
            float o[D / 8][4];
#pragma unroll
            for (int n = 0; n < D / 8; ++n) { o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f; }
            float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f}, r_run[2] = {-INFINITY, -INFINITY};
            for (int t = 0; t < w.n_tiles && ok; ++t) {
                if (!mbar_wait_warp(&full_bar[s], ph, abort_ptr)) { ok = false; break; }
                attend_tile<D, MT, TS, TILE>(p, w.b, w.g, w.L, w.c_end, w.c_begin + t * TILE, smem + (size_t)s * Cfg::kStageBytes, q_base, no_q, mt, ts,
                                             lane, j0, j1, scale_log2, [&](int pos) { return p.page_table[(size_t)w.b * p.max_pages + pos / kPageSize]; },
                                             o, m_run, l_run, r_run);
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty_bar[s]);
                if (++s == E) { s = 0; ph ^= 1u; }
            }
            settle<D>(o, m_run, r_run);
            l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 1);
            l_run[0] += __shfl_xor_sync(0xffffffffu, l_run[0], 2);
            l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 1);
            l_run[1] += __shfl_xor_sync(0xffffffffu, l_run[1], 2);
            if ((lane & 3) == 0) {
                s_m[warp][lane >> 2] = m_run[0]; s_l[warp][lane >> 2] = l_run[0];
                s_m[warp][(lane >> 2) + 8] = m_run[1]; s_l[warp][(lane >> 2) + 8] = l_run[1];
            }
            sync_warps();                      // the query rows have been read: their space carries the exchange
            // the second warp of a row group hands its accumulator over, half of the columns at a time
            float own[2], other[2], M[2];
            {
                const int peer = warp ^ 1;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = (lane >> 2) + 8 * h;
                    const float mo = s_m[peer][r];
                    M[h] = fmaxf(m_run[h], mo);
                    own[h] = m_run[h] == -INFINITY ? 0.f : exp2f(m_run[h] - M[h]);
                    other[h] = mo == -INFINITY ? 0.f : exp2f(mo - M[h]);
                    l_run[h] = l_run[h] * own[h] + s_l[peer][r] * other[h];
                }
            }
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                if (ts == 1) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const int n = half * (D / 16) + k;
                        exchange[k * 32] = make_float4(o[n][0], o[n][1], o[n][2], o[n][3]);
                    }
                }
                sync_warps();
                if (ts == 0) {
#pragma unroll
                    for (int k = 0; k < D / 16; ++k) {
                        const int n = half * (D / 16) + k;
                        const float4 v = exchange[k * 32];
                        o[n][0] = o[n][0] * own[0] + v.x * other[0]; o[n][1] = o[n][1] * own[0] + v.y * other[0];
                        o[n][2] = o[n][2] * own[1] + v.z * other[1]; o[n][3] = o[n][3] * own[1] + v.w * other[1];
                    }
                }
                sync_warps();
            }
            if (ts != 0 || mt * 16 >= rows || !ok) continue;
            if (!w.whole) {
                // unit (mt * D/8 + n) * 32 + lane of the piece: (row r0: columns c, c+1; row r1: the same), c = 8 n + 2 (lane % 4)
                size_t at = slot;
                if (!MASSV_IN_BOUNDS(at, 2 * kFlatMaxCtas, p.dev_status)) at = 0;
                float4* dst = reinterpret_cast<float4*>(p.flat_part_o + at * RP * D) + mt * (D / 8) * 32 + lane;
#pragma unroll
                for (int n = 0; n < D / 8; ++n) dst[n * 32] = make_float4(o[n][0], o[n][1], o[n][2], o[n][3]);
                if ((lane & 3) == 0) {
                    float2* ml = reinterpret_cast<float2*>(p.flat_part_ml + at * RP * 2);
                    ml[r0] = make_float2(M[0], l_run[0]);
                    ml[r1] = make_float2(M[1], l_run[1]);
                }
            } else {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int r = h ? r1 : r0;
                    if (r >= rows) continue;
                    const size_t row_out = ((size_t)w.b * p.R + r / G) * p.Hq + w.g * G + r % G;
                    const float inv = 1.f / l_run[h];
#pragma unroll
                    for (int n = 0; n < D / 8; ++n) {
                        const float x = o[n][2 * h] * inv, y = o[n][2 * h + 1] * inv;
                        const size_t at = row_out * D + n * 8 + 2 * (lane & 3);
                        *reinterpret_cast<uint32_t*>(p.out + at) = pack_bf16(x, y);
                        if (p.out_f32) *reinterpret_cast<float2*>(p.out_f32 + at) = make_float2(x, y);
                    }
                    if (p.lse && (lane & 3) == 0) p.lse[row_out] = (M[h] + log2f(l_run[h])) * 0.6931471805599453f;
                }
            }
        }
    }
    pdl_trigger();
    __syncthreads();
    if (threadIdx.x == 0 && abort_flag) set_status(p.dev_status, MASSV_ERR_TIMEOUT);
}

// Merge the chunks of sequences that span more than one: one CTA per
// (sequence, KV head, query row), one thread per channel.
constexpr int kCombineMaxChunks = 1024;
__global__ void __launch_bounds__(128) attn_combine_kernel(const AttnParams p, int rows_pad) {
    const int G = p.Hq / p.Hkv, rows = G * p.R;
    const int r = blockIdx.x % rows, g = (blockIdx.x / rows) % p.Hkv, b = blockIdx.x / (rows * p.Hkv);
    pdl_wait();
    pdl_trigger();
    const int L = p.seq_lens[b];
    if (L < 0 || L + p.R > p.max_pages * kPageSize) return;
    const int first_chunk = (p.window > 0 ? max(0, L - p.window + 1) : 0) / p.kv_chunk;   // as in the split kernel
    const int n_chunks = (L + p.R + p.kv_chunk - 1) / p.kv_chunk - first_chunk;
    if (n_chunks <= 1) return;
    __shared__ float s_w[kCombineMaxChunks];    // first the chunk maxima, then the merge weights
    __shared__ float s_l[kCombineMaxChunks];
    const size_t item0 = ((size_t)b * p.Hkv + g) * p.max_chunks + first_chunk;
    for (int c = threadIdx.x; c < n_chunks; c += blockDim.x) {
        const float2 ml = *reinterpret_cast<const float2*>(p.part_ml + ((item0 + c) * rows_pad + r) * 2);
        s_w[c] = ml.x;
        s_l[c] = ml.y;
    }
    __syncthreads();
    float M = -INFINITY;
    for (int c = 0; c < n_chunks; ++c) M = fmaxf(M, s_w[c]);
    __syncthreads();
    for (int c = threadIdx.x; c < n_chunks; c += blockDim.x) s_w[c] = s_w[c] == -INFINITY ? 0.f : exp2f(s_w[c] - M);
    __syncthreads();
    float Lsum = 0.f;
    for (int c = 0; c < n_chunks; ++c) Lsum += s_l[c] * s_w[c];
    const float inv = 1.f / Lsum;
    const int j = r / G, hh = r % G;
    const size_t row_out = ((size_t)b * p.R + j) * p.Hq + g * G + hh;
    const float* src = p.part_o + (item0 * rows_pad + r) * p.d;
    const size_t chunk_stride = (size_t)rows_pad * p.d;
    for (int col = threadIdx.x; col < p.d; col += blockDim.x) {
        float acc = 0.f;
        int c = 0;
        for (; c + 4 <= n_chunks; c += 4) {      // four independent loads in flight, summed in chunk order
            const float v0 = src[(size_t)c * chunk_stride + col], v1 = src[(size_t)(c + 1) * chunk_stride + col];
            const float v2 = src[(size_t)(c + 2) * chunk_stride + col], v3 = src[(size_t)(c + 3) * chunk_stride + col];
            acc += v0 * s_w[c]; acc += v1 * s_w[c + 1]; acc += v2 * s_w[c + 2]; acc += v3 * s_w[c + 3];
        }
        for (; c < n_chunks; ++c) acc += src[(size_t)c * chunk_stride + col] * s_w[c];
        acc *= inv;
        p.out[row_out * p.d + col] = __float2bfloat16(acc);
        if (p.out_f32) p.out_f32[row_out * p.d + col] = acc;
    }
    if (p.lse && threadIdx.x == 0) p.lse[row_out] = (M + log2f(Lsum)) * 0.6931471805599453f;
}

template <int D, int MT, int TS, int TILE>
cudaError_t launch_split(const AttnParams& p, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t stream) {
    using Cfg = AttnCfg<D, TILE, (MT * TS + 1 > 4)>;
    constexpr int RP = MT * 16;
    const size_t ring = (size_t)Cfg::kStages * Cfg::kStageBytes;
    static_assert((size_t)TS * RP * D * 4 + 2 * TS * RP * 4 <= (size_t)Cfg::kStages * Cfg::kStageBytes, "merge staging fits the ring");
    const size_t smem = ring + (size_t)RP * D * 2 + 1024;
    cudaError_t e = cudaFuncSetAttribute(attn_split_kernel<D, MT, TS, TILE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(attn_split_kernel<D, MT, TS, TILE>, dim3(p.max_chunks, p.Hkv, p.B), dim3((MT * TS + 1) * 32), smem, stream, mk, mv, p);
}

template <int D, int MT, int TILE>
cudaError_t launch_flat(const AttnParams& p, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t stream, int* ctas) {
    using Cfg = FlatCfg<D, MT, TILE>;
    const size_t smem = (size_t)Cfg::kSmem + (size_t)(p.B + 1) * sizeof(int);
    // (The attribute is the process's, not the call's: every call sets the same bound, so that a small batch on one thread cannot
    // lower it between another thread's attribute and launch.)
    constexpr int kMaxSmem = Cfg::kSmem + (kFlatMaxBatchMeta + 1) * (int)sizeof(int);
    static_assert(kMaxSmem <= 225 * 1024, "ring, query rows and tile counts fit shared memory");
    *ctas = device_sm_count() * Cfg::kCtasPerSm;
    if (*ctas > kFlatMaxCtas) *ctas = kFlatMaxCtas;
    // A range is no longer than pairs / CTAs of the longest pair, which has at least kPairUnits + 1 units: with 3 pairs or fewer for 5 CTAs no
    // lengths meet flat_range's condition for a pair per CTA, with more pairs than CTAs none can.
    const long pairs = (long)p.B * p.Hkv;
    const bool whole = pairs <= *ctas && 5 * pairs > 3L * *ctas;
    const auto kernel = whole ? attn_flat_kernel<D, MT, TILE, true> : attn_flat_kernel<D, MT, TILE, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
    if (e != cudaSuccess) return e;
    // the query rows as a [B * R * Hq, D] matrix; a box is the G adjacent heads of one block row
    CUtensorMap mq;
    if (!make_tensor_map_bf16_2d(&mq, p.q, (uint64_t)p.B * p.R * p.Hq, D, (uint32_t)(p.Hq / p.Hkv))) return cudaErrorInvalidValue;
    return launch_pdl(kernel, dim3(*ctas), dim3((Cfg::kWarps + 1) * 32), smem, stream, mk, mv, mq, p);
}

template <int D>
cudaError_t launch_split_d(const AttnParams& p, int mt, const CUtensorMap& mk, const CUtensorMap& mv, cudaStream_t stream) {
    switch (mt) {
        // d = 256 uses 32-token stages so that two CTAs (three 32 KB stages each) share an SM and
        // one CTA's set-up and merge overlap the other's streaming
        case 1: return D == 256 ? launch_split<D, 1, 2, 32>(p, mk, mv, stream) : launch_split<D, 1, 2, 64>(p, mk, mv, stream);
        case 2: return D == 256 ? launch_split<D, 2, 1, 32>(p, mk, mv, stream) : launch_split<D, 2, 1, 64>(p, mk, mv, stream);
        case 3: return D == 256 ? launch_split<D, 3, 1, 32>(p, mk, mv, stream) : launch_split<D, 3, 1, 64>(p, mk, mv, stream);
        case 4: return D == 256 ? launch_split<D, 4, 1, 32>(p, mk, mv, stream) : launch_split<D, 4, 1, 64>(p, mk, mv, stream);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

int attn_rows_pad(int group_rows) { return (group_rows + 15) / 16 * 16; }

// Which split kernel runs.  The warp-MMA kernel re-reads every K/V tile from shared memory once
// per 16 query rows, which saturates the shared-memory pipe from about 48 rows up; the tcgen05
// kernel reads each tile once whatever the row count, and with its balanced schedule it is the
// faster one on every head_dim <= 128 shape measured.  At head_dim 256 its ring leaves room for one
// CTA per SM only, and the warp-MMA kernel (few rows per KV head on such models) stays ahead.
bool attn_use_umma(const AttnParams& p) {
    if (p.path == 1 || !attn_umma_supported(p)) return false;
    if (p.path == 2) return true;
    return p.d <= 128;
}

// The most positions a (sequence, KV head) pair can need.
static long pair_tokens(const AttnParams& p) {
    const long tokens = (long)p.max_pages * kPageSize, seen = (long)p.window + p.R + 64;       // (a window may be any int32)
    return p.window > 0 && seen < tokens ? seen : tokens;
}

// tcgen05 kernel: one CTA per pair where pairs are short, instead of ranges of the line of tiles: nothing to deal out, no pieces and
// no merge launch.  A CTA takes 6 - 7.5 us and 1.2 - 1.5 us per tile of 64 positions, the balanced line with its merge at least
// 9 - 10 us and more the more pairs it cuts.  The bounds are where full tables and lengths from a quarter of the table up, 1 and 42
// rows, are all no slower this way (tables of 1 - 10 tiles, 44 batches, both head_dims).  Call times, balanced -> one CTA per pair, head_dim 128:
//   1 x 4 pairs     2 tiles 10.4 -> 7.9 us    3 tiles 11.0 -> 9.0     4 tiles, full 11.4 -> 12.1
//   16 x 4          2 tiles 13.8 -> 9.3       5 tiles 14.8 -> 13.9    6 tiles, full, 1 row 1.08 of the time
//   32 x 4          7 tiles, full 23.5 -> 16.9                        8 tiles, full, 1 row 1.05
//   32 x 8          3 tiles 15.1 -> 12.3      8 tiles 29.8 -> 20.2
// and head_dim 64, whose CTAs are shorter: 16 x 4 of 6 tiles 13.4 -> 12.7, of 7, full, 1.06; 24 x 4 of 8 17.0 -> 15.2, of 9 14.7 -> 16.4.
// With more pairs than places for CTAs (two on an SM) there is a second wave, and full tables of which the line takes whole pairs per
// range cut nothing there: 64 x 8 of 4 tiles 33.7 -> 26.4, of 8 47.7 -> 40.2, but of 3 (six tiles a range) 20.9 -> 23.1; 38 x 8 of 6 tiles
// 30.6 -> 30.4, of 7 31.5 -> 33.4; from two waves on few pairs are cut (80 x 8 of 8 full 53.0 -> 57.3), though ragged lengths still gain.
static bool one_piece_per_pair(const AttnParams& p) {
    if (p.chunk_forced || p.d > 128 || p.max_pages > kMaxChunkPages) return false;
    const long pairs = (long)p.B * p.Hkv, tiles = (pair_tokens(p) + 63) / 64, slots = 2L * device_sm_count();
    if (pairs <= slots) {
        if (p.d == 64) return tiles <= (pairs < 8 ? 3 : 4) + (pairs < 96 ? pairs / 24 : 4);
        return tiles <= (pairs < 16 ? 3 : pairs < 48 ? 4 : pairs < 128 ? 5 : pairs < 192 ? 7 : 8);
    }
    const long range = (pairs * tiles + slots - 1) / slots;          // tiles of the line per CTA
    return pairs <= 2 * slots && tiles >= 3 && tiles <= (2 * pairs < 3 * slots ? 6 : 8) && range % tiles != 0;
}

// Balanced schedule or chunk grid for the warp-MMA kernel at head_dim 256.  The balanced one wins wherever the grid would cut
// a pair into chunks, since that costs CTAs that retire at once and a merge as well (times of a call, page table for 8,192
// positions: 32 x 8 pairs of 2k - 8k positions 243 -> 224 us, of 100 - 900 50 -> 38, of 1 - 100 24 -> 23; a window of 1,024 on long
// contexts 79 -> 62; 2 x 8 pairs of 1,000 positions 18.5 -> 16.6).  Where the table holds no more than one chunk, a grid of
// one-pair CTAs has no ranges to cut and nothing to merge: it wins as long as its CTAs are resident at once (30 x 8 pairs of
// 1 - 104 positions 17 against 23 us, of 400 - 600 34 against 38; 18 x 8 of 160 - 312 19 against 23), and up to about 544 positions
// beyond that (64 x 8 pairs of 1 - 184: 35 against 37, of 272 - 536: 59 against 57, of 600 - 792: 89 against 81).  From 17
// query rows up the balanced kernel's two warps per row group decide it (24 x 8 pairs of 24 rows, 1 - 54 positions: 33 -> 20 us;
// 64 x 4 pairs of 36 rows, 2k - 6k: 412 -> 268).
static bool use_flat_warp_mma(const AttnParams& p, int mt) {
    if (p.d != 256 || p.chunk_forced || p.B > kFlatMaxBatchMeta) return false;
    if (mt > 1 || p.max_chunks > 1) return true;
    return pair_tokens(p) > 544 && (long)p.B * p.Hkv > 2L * device_sm_count();
}

cudaError_t launch_verify_attn(const AttnParams& p, cudaStream_t stream) {
    if (p.kv_chunk % kChunkAlign != 0 || p.kv_chunk > kMaxChunkPages * kPageSize) return cudaErrorInvalidValue;
    CUtensorMap mk, mv;
    const uint64_t rows_total = (uint64_t)p.num_pages * p.Hkv * kPageSize;
    if (!make_tensor_map_bf16_2d(&mk, p.k_pages, rows_total, p.d, kPageSize) ||
        !make_tensor_map_bf16_2d(&mv, p.v_pages, rows_total, p.d, kPageSize))
        return cudaErrorInvalidValue;
    const int rows = (p.Hq / p.Hkv) * p.R;
    const int mt = attn_rows_pad(rows) / 16;
    cudaError_t e;
    const TimingHooks& hooks = timing_hooks();
    if (hooks.attn_start && cudaEventRecord(hooks.attn_start, stream) != cudaSuccess) return cudaGetLastError();
    if (attn_use_umma(p)) {
        const bool one_piece = one_piece_per_pair(p), flat = !one_piece && !p.chunk_forced && attn_umma_flat_supported(p);
        int launched = 0;
        if (one_piece) {
            AttnParams q = p;
            q.kv_chunk = (p.max_pages * kPageSize + kChunkAlign - 1) / kChunkAlign * kChunkAlign;
            q.max_chunks = 1;
            q.follow_tiles = true;
            e = launch_attn_umma(q, mk, mv, stream, false, &launched, nullptr);
            if (e != cudaSuccess) return e;
            if (hooks.attn_stop && cudaEventRecord(hooks.attn_stop, stream) != cudaSuccess) return cudaGetLastError();
            count_launches(launched);
            return cudaGetLastError();
        }
        e = launch_attn_umma(p, mk, mv, stream, flat, &launched, hooks.attn_stop);
        if (e != cudaSuccess) return e;
        if (flat) {
            count_launches(launched);
            return cudaGetLastError();
        }
    } else if (use_flat_warp_mma(p, mt)) {
        int ctas = 0;
        switch (mt) {
            case 1: e = launch_flat<256, 1, 32>(p, mk, mv, stream, &ctas); break;
            case 2: e = launch_flat<256, 2, 32>(p, mk, mv, stream, &ctas); break;
            case 3: e = launch_flat<256, 3, 32>(p, mk, mv, stream, &ctas); break;
            case 4: e = launch_flat<256, 4, 32>(p, mk, mv, stream, &ctas); break;
            default: return cudaErrorInvalidValue;
        }
        if (e != cudaSuccess) return e;
        if (hooks.attn_stop && cudaEventRecord(hooks.attn_stop, stream) != cudaSuccess) return cudaGetLastError();
        e = launch_flat_combine(p, ctas, stream);
        if (e != cudaSuccess) return e;
        count_launches(2);
        return cudaGetLastError();
    } else {
        switch (p.d) {
            case 64: e = launch_split_d<64>(p, mt, mk, mv, stream); break;
            case 128: e = launch_split_d<128>(p, mt, mk, mv, stream); break;
            case 256: e = launch_split_d<256>(p, mt, mk, mv, stream); break;
            default: return cudaErrorInvalidValue;
        }
    }
    if (e != cudaSuccess) return e;
    if (hooks.attn_stop && cudaEventRecord(hooks.attn_stop, stream) != cudaSuccess) return cudaGetLastError();
    int launched = 1;
    if (p.max_chunks > 1) {
        if (p.max_chunks > kCombineMaxChunks) return cudaErrorInvalidValue;
        e = launch_pdl(attn_combine_kernel, dim3(p.B * p.Hkv * rows), dim3(p.d < 128 ? 64 : 128), 0, stream, p, attn_rows_pad(rows));
        if (e != cudaSuccess) return e;
        launched = 2;
    }
    count_launches(launched);
    return cudaGetLastError();
}

}  // namespace massv
