// Base-weight GEMM fused with the SALT delta (Section "Multi-Tenant Serving":
// the served weight is W_final = W_base + gamma * Wbar + delta_i).  For one
// projection:
//
//     y[t, :] = x[t, :] W_base + s_c (x[t] A_c) B_c + s_u (x[t] a_u) b_u
//
// y is written, never read.  The low-rank part reuses the apply path's row
// blocks: a shrink-only launch of the apply kernel leaves every block's V_ext
// tile (scaled and masked as in the apply) in the segments workspace; this
// kernel runs the GEMM over tiles of tokens in grouped order and, for every
// row block overlapping a tile, adds V_ext * Stack_B into the same
// tensor-memory accumulator: further K chunks whose A operand holds the
// block's V rows at their tile rows and zeros elsewhere, and whose MMAs leave
// the other rows' lanes alone.  Tokens with no term are in no block and get
// x W_base alone.
//
// CG = 2 (batches of more than 128 tokens): a cluster of two CTAs computes a
// 256-token x BN tile with cta_group::2 MMAs.  Each CTA loads its own 128
// token rows and half of the W columns, so a 64-wide K chunk moves 32 KB into
// each SM per 512 tensor cycles at BN = 256 (a 128 x 128 tile of one CTA
// moves the same per 256, which bound the GEMM on L2-to-SM traffic).
// CG = 1 (up to 128 tokens): one CTA, 128 x BN; only the batch's rows are
// loaded, the tile is bound by streaming W.
//
// Persistent CTAs over units (tile, K split of KS).  Warp roles:
//   warp 0      TMA of the W tile (either layout lands as its UMMA descriptor
//               reads it), and of x where a tile's rows are consecutive
//               tokens;
//   warp 1      tcgen05.mma into one of two BN-column accumulators;
//   warps 2-7   everything gathered, by cp.async, a whole stage a warp (six
//               stages in flight): the token rows of a K chunk, or a delta
//               chunk's V rows and stacked B rows;
//   warps 8-11  epilogue: fp32 -> bf16 (RNE) and store, one token row a
//               thread; with K splits the fp32 partials go through the
//               workspace and are summed in split order (so the result does
//               not depend on timing).
// The launch is a programmatic dependent of the shrink, which releases it
// once everything before the shrink is complete: the K loop over x and W
// overlaps the shrink's tail, and only the delta and the partial stores wait
// for the shrink itself.
//
// Measured against one CTA per 128 x 128 tile with cp.async for x, no K
// split and the shrink run to its end first: a 3B MLP layer at 8192 tokens
// 2939 -> 882 us (1.42 PFLOP/s), an 8B layer at 512 tokens 748 -> 322 us, at
// 24 tokens 551 -> 175 us; single calls of 1 to 4096 tokens, 256 to 8192 wide,
// 1.14 (4096 x 512 x 512) to 5.0 times as fast.  x by TMA tile::gather4 instead of the gather
// warps took 3050 us for the first (about 90 cycles a four-row copy).
#include <cuda_bf16.h>

#include <algorithm>

#include "salt_async.cuh"
#include "salt_internal.cuh"
#include "salt_pipe.cuh"
#include "salt_tcgen05.cuh"

namespace salt {
namespace {

constexpr int BM = 128;                    // token rows per CTA (the UMMA M is BM * CG)
constexpr int BK = 64;                     // K chunk (128-byte rows)
constexpr int NST_MAX = 10;
constexpr int BASE_RING = 224 * 1024;      // shared-memory ring: 7 stages of a 256-column pair tile
constexpr int BASE_THREADS = 384;
constexpr int GW0 = 2, GWN = 6;            // gather warps; the ring holds at least as many stages (below)
constexpr int EW0 = 8;                     // first epilogue warp
constexpr int EPI_N = 128;
constexpr int BAR_E = 1;                   // named barrier of the epilogue warps
constexpr int MT_MAX = SALT_MAX_TOKENS / (2 * BM);  // M tiles (of pairs: batches of one tile take CG = 1)
constexpr int BASE_KS_MAX = 16;
constexpr int SPLIT_POLLS = 128;           // a split's wait for the others of its tile
static_assert(BASE_KS_MAX <= 16, "a split is a bit of half a counter word");

struct BaseInfo {
    uint64_t full[NST_MAX], empty[NST_MAX];
    uint64_t accf[2], acce[2];
    int32_t mt_b0[MT_MAX], mt_b1[MT_MAX];  // row blocks overlapping M tile: [b0, b1)
    uint32_t mt_nd[MT_MAX / 2];            // its delta chunks (at most 512), two tiles to a word
    uint16_t mt_x0[MT_MAX];                // its first token, X_GATHER and X_PEER
    uint32_t tmem;
    uint32_t shares;
    uint32_t dstage[NST_MAX];              // a delta stage: its K = 16 steps, first and end row of its block in the tile (10 bits each)
    alignas(16) uint32_t token[4];         // copied by the second CTA's gather warps to signal the first
};
constexpr size_t BASE_SMEM = 1024 + BASE_RING + (sizeof(BaseInfo) + 15) / 16 * 16;
// (an SM has 228 KB, of which it keeps 1 KB a CTA: room for a swap CTA beside)
static_assert(BASE_SMEM + 2 * 1024 <= 228 * 1024, "shared memory exceeds what an SM has beside a swap CTA");
constexpr uint16_t X_GATHER = 1u << 15;  // this CTA's rows of the tile are not consecutive tokens
constexpr uint16_t X_PEER = 1u << 14;    // the pair's second CTA's are not
static_assert(SALT_MAX_TOKENS <= X_PEER, "mt_x0 holds a token index below the flags");
// A gather warp fills every GWN-th stage and waits only for its own slots'
// phases; with at least GWN stages a slot's barrier is never two phases
// behind the one it waits for (a parity wait could not tell).
static_assert(BASE_RING / (2 * BM * 128) >= GWN, "stages for the gather warps");

__device__ __forceinline__ const uint16_t *res_b_row(const BaseParams &p, int e)
{
    const int slot = res_slot(e), rank = res_rank(e), k = res_k(e);
    const uint16_t *base = reinterpret_cast<const uint16_t *>(p.pool + (int64_t)slot * p.slot_stride +
                                                              SALT_BLOB_HEADER_BYTES) + (int64_t)rank * p.res_off;
    return base + (int64_t)rank * p.d_in + (int64_t)k * p.d_out;
}

// 32 consecutive bytes of an output row
__device__ __forceinline__ void store32(uint16_t *dst, const uint32_t (&w)[8], bool wide)
{
    if (wide) {
        asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]),
                     "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
    } else {
        *reinterpret_cast<uint4 *>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4 *>(dst + 8) = make_uint4(w[4], w[5], w[6], w[7]);
    }
}
__device__ __forceinline__ void store_part8(float *dst, const uint32_t *v)
{
    asm volatile("st.global.cg.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]),
                 "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                 : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
}

// A position in the ring of n stages and its phase parity.
struct RingPos {
    uint32_t slot = 0, phase = 0;
    __device__ __forceinline__ void advance(uint32_t by, uint32_t n)
    {
        for (slot += by; slot >= n; slot -= n) phase ^= 1u;
    }
};

template <int CG>
__global__ void __launch_bounds__(BASE_THREADS, 1) salt_base_kernel(const __grid_constant__ BaseParams p)
{
    extern __shared__ __align__(128) uint8_t smem_raw[];
    uint8_t *ring = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
    BaseInfo &info = *reinterpret_cast<BaseInfo *>(ring + BASE_RING);
    const uint32_t ring32 = smem_u32(ring);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = CG == 2 ? (int)cluster_ctarank() : 0;  // this CTA's half of the tile
    const int cl = blockIdx.x / CG, n_cl = gridDim.x / CG;
    // The batch as built last: a captured launch is replayed on later ones.
    // The launch is shaped for up to p.T tokens; of more it computes nothing.
    const int T = p.counts[0] <= p.T ? p.counts[0] : 0;
    const int BN = p.bn, NB = BN / CG;                      // NB: W columns this CTA loads
    const int n_mt = (T + BM * CG - 1) / (BM * CG), n_nt = (p.d_out + BN - 1) / BN;
    const int KS = p.ks, n_units = n_mt * n_nt * KS;
    const int nk = (p.d_in + BK - 1) / BK;
    // a stage: the CTA's token rows (only as many as the batch can fill),
    // then its W columns.  The UMMA reads 128 rows: with fewer loaded the
    // rest are whatever follows, and reach only accumulator rows past T.
    const int m_rows = CG == 2 ? BM : (min(p.T, BM) + 15) & ~15;
    const uint32_t x_bytes = (uint32_t)m_rows * 128u, stage = x_bytes + (uint32_t)NB * 128u;
    const uint32_t nst = min((uint32_t)NST_MAX, (uint32_t)BASE_RING / stage);
    auto bar = [](const uint64_t &b) { return smem_u32(&b); };

    pdl_launch_dependents();
    if (warp == 1) {
        tmem_alloc<CG>(smem_u32(&info.tmem), 2 * BN);
        tmem_relinquish<CG>();
    }
    if (p.counts[0] > p.T && blockIdx.x == 0 && tid == 0) atomicOr(p.err, SALT_DEVERR_BATCH);
    if (tid == 0) {
        for (int i = 0; i < NST_MAX; ++i) {
            mbar_init(bar(info.full[i]), 1 + CG);  // the TMA warps and the first CTA's gather warp
            mbar_init(bar(info.empty[i]), 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(info.accf[i]), 1);
            mbar_init(bar(info.acce[i]), 4 * CG);
        }
        mbar_fence_init();
    }
    for (int i = tid; i < n_mt; i += BASE_THREADS) {
        info.mt_b0[i] = 0x7fffffff;
        info.mt_b1[i] = 0;
        info.mt_nd[i >> 1] = 0;
    }
    __syncthreads();
    // Row blocks lie in grouped order and hold at most TM tokens, so each
    // overlaps one or two M tiles.  (The segment tables are complete: they
    // were written before the shrink started.)
    const int n_blk = min(p.counts[3], p.blk_cap);
    for (int b = tid; b < n_blk; b += BASE_THREADS) {
        const int4 r = *reinterpret_cast<const int4 *>(p.blk + BLK_INTS * b);
        const int S = r.w + p.blk[BLK_INTS * b + BLK_NRES];
        if (S <= 0 || S > S_MAX || r.y <= 0) continue;  // flagged by the shrink
        const int t0 = r.x / (BM * CG), t1 = min((r.x + r.y - 1) / (BM * CG), n_mt - 1);
        for (int t = t0; t <= t1; ++t) {
            atomicMin(&info.mt_b0[t], b);
            atomicMax(&info.mt_b1[t], b + 1);
            atomicAdd(&info.mt_nd[t >> 1], (uint32_t)((S + BK - 1) / BK) << (16 * (t & 1)));
        }
    }
    // Tiles whose rows are consecutive tokens (runs of a prefill batch) take x
    // by plain TMA tiles; a batch of one tile is not looked at.
    for (int t = warp; t < n_mt; t += BASE_THREADS / 32) {
        uint32_t x = 0;
        for (int h = rank; h < CG; ++h) {  // the first CTA looks at both halves
            const int m0 = (t * CG + h) * BM, rows = min(BM, T - m0);
            bool lin = CG == 2 && rows > 0;
            const int x0 = lin ? p.perm[m0] : 0;
            for (int i = lane; i < rows && lin; i += 32) lin = p.perm[m0 + i] == x0 + i;
            lin = __all_sync(0xffffffffu, lin);
            if (h == rank) x |= lin ? (uint32_t)x0 : X_GATHER;
            if (h == 1 && !lin) x |= X_PEER;
        }
        if (lane == 0) info.mt_x0[t] = (uint16_t)x;
    }
    tc_fence_before();
    cta_or_cluster_sync<CG>();
    tc_fence_after();
    const uint32_t tmem = info.tmem;
    bool ok = true;  // a bounded wait gave up: no further waits, no further loads
    auto wait_bar = [&](const uint64_t &b, uint32_t parity) {
        if (ok && !mbar_wait(smem_u32(&b), parity)) ok = false;
    };
    // a stage; peer: a thread of the pair's second CTA staged some of it
    auto wait_full = [&](uint32_t slot, uint32_t parity, bool peer) {
        const uint32_t b = smem_u32(&info.full[slot]);
        if (ok && !(peer ? mbar_wait_cluster<CG>(b, parity) : mbar_wait(b, parity))) ok = false;
    };
    // unit u: tile u / KS (M tile tile % n_mt: the M tiles of one W column
    // block run side by side, so W is read from memory about once), split u % KS
    auto chunk_lo = [&](int s) { return nk * s / KS; };
    const bool in_out = p.w_layout == SALT_W_IN_OUT;
    auto n_delta = [&](int mt, int s) {
        const int nd = (int)(info.mt_nd[mt >> 1] >> (16 * (mt & 1)) & 0xffffu);
        return nd > s ? (nd - s + KS - 1) / KS : 0;
    };

    if (warp == 0) {
        // ============================================================ TMA
        RingPos rp;
        bool wrapped = false;  // the ring's first round needs no wait
        auto next_slot = [&]() {
            if (wrapped) wait_bar(info.empty[rp.slot], rp.phase ^ 1u);
            ok = __all_sync(0xffffffffu, ok);
        };
        auto advance = [&]() {
            rp.advance(1, nst);
            wrapped = wrapped || rp.slot == 0;
        };
        for (int u = cl; u < n_units && ok; u += n_cl) {
            const int tile = u / KS, s = u - tile * KS, mt = tile % n_mt, n0 = tile / n_mt * BN + rank * NB;
            const int k1 = chunk_lo(s + 1), xt = info.mt_x0[mt], x0 = xt & (X_PEER - 1);
            const bool lin = !(xt & X_GATHER), peer = CG == 2 && rank == 0 && (xt & X_PEER);
            for (int kc = chunk_lo(s); kc < k1 && ok; ++kc, advance()) {
                next_slot();
                if (!ok) break;
                if (elect_one()) {
                    const uint32_t ws = ring32 + rp.slot * stage + x_bytes;
                    const uint32_t fb = leader_addr<CG>(bar(info.full[rp.slot]));
                    const int k0 = kc * BK;
                    mbar_expect_tx_cluster<CG>(fb, (uint32_t)NB * 128u + (lin ? x_bytes : 0u) + (peer ? BULK_SIGNAL_BYTES : 0u));
                    if (lin) tma_load_2d_cg<CG>(ws - x_bytes, &p.xmap, k0, x0, fb);
                    if (in_out) {
                        // W[d_in][d_out]: boxes of 64 K rows x 64 N columns (MN-major)
                        for (int h = 0; h < NB / 64; ++h) tma_load_2d_cg<CG>(ws + h * 8192, &p.wmap, n0 + 64 * h, k0, fb);
                    } else {
                        // W[d_out][d_in]: one box of NB rows x 64 K (K-major)
                        tma_load_2d_cg<CG>(ws, &p.wmap, k0, n0, fb);
                    }
                }
                __syncwarp();
            }
            // the delta's stages hold nothing of W
            for (int j = n_delta(mt, s); j > 0 && ok; --j, advance()) {
                next_slot();
                if (ok && elect_one()) {
                    const uint32_t fb = leader_addr<CG>(bar(info.full[rp.slot]));
                    if (CG == 2 && rank == 0) mbar_expect_tx_cluster<CG>(fb, BULK_SIGNAL_BYTES);
                    else mbar_arrive_relaxed_cluster<CG>(fb);
                }
                __syncwarp();
            }
        }
        // every stage released (with CG = 2 by the pair's first CTA, whose
        // arrivals must find this CTA's barriers alive)
        for (uint32_t i = 0; i < nst; ++i, advance())
            if (wrapped) wait_bar(info.empty[rp.slot], rp.phase ^ 1u);
    } else if (warp == 1) {
        // ============================================================ MMA issue
        if (rank == 0) {
            const uint32_t id_k = idesc_bf16_f32(BM * CG, BN), id_mn = idesc_bf16_f32_bmn(BM * CG, BN);
            // descriptors of the ring's first stage; a stage adds stage / 16, a
            // K step 2 (K-major: 32 bytes) or 128 (MN-major: 16 rows)
            const uint64_t x0 = sdesc_kmajor_sw128(ring32), wk0 = sdesc_kmajor_sw128(ring32 + x_bytes);
            const uint64_t wmn0 = sdesc_mnmajor_sw128_lbo(ring32 + x_bytes, 8192);
            const uint32_t st16 = stage >> 4;
            const uint64_t w0 = in_out ? wmn0 : wk0;
            const uint32_t w_step = in_out ? 128 : 2, id_w = in_out ? id_mn : id_k;
            RingPos rp;
            uint32_t lt = 0;
            for (int u = cl; u < n_units; u += n_cl, ++lt) {
                const int tile = u / KS, s = u - tile * KS, mt = tile % n_mt;
                const uint32_t buf = lt & 1, acc = tmem + buf * BN;
                if (lt >= 2) wait_bar(info.acce[buf], ((lt - 2) >> 1) & 1);
                tc_fence_after();
                uint32_t accum = 0;
                const bool peer = CG == 2 && (info.mt_x0[mt] & X_PEER);
                for (int n = chunk_lo(s + 1) - chunk_lo(s); n > 0; --n, rp.advance(1, nst)) {
                    wait_full(rp.slot, rp.phase, peer);
                    tc_fence_after();
                    const uint64_t xd = x0 + rp.slot * st16, wd = w0 + rp.slot * st16;
                    if (elect_one()) {
#pragma unroll
                        for (int kk = 0; kk < BK / 16; ++kk)
                            umma_bf16_cg<CG>(acc, xd + kk * 2, wd + kk * w_step, id_w, kk > 0 ? 1u : accum);
                        umma_commit_cg<CG>(bar(info.empty[rp.slot]));
                    }
                    __syncwarp();
                    accum = 1;
                }
                // (added to at least one K chunk's product: KS <= nk)
                for (int n = n_delta(mt, s); n > 0; --n, rp.advance(1, nst)) {
                    wait_full(rp.slot, rp.phase, CG == 2);
                    tc_fence_after();
                    const uint64_t xd = x0 + rp.slot * st16, wd = wmn0 + rp.slot * st16;
                    ok = __all_sync(0xffffffffu, ok);
                    // only the block's own rows: an infinity in its B times the
                    // other rows' zeros would be a NaN in theirs
                    const uint32_t ds = ok ? *reinterpret_cast<volatile uint32_t *>(&info.dstage[rp.slot]) : 0u;
                    const int steps = (int)(ds & 0x3ffu);
                    uint32_t off[4 * CG];
                    lanes_off<CG>((int)(ds >> 10 & 0x3ffu), (int)(ds >> 20), off);
                    if (elect_one()) {
                        for (int kk = 0; kk < steps; ++kk)
                            umma_bf16_cg_lanes<CG>(acc, xd + kk * 2, wd + kk * 128, id_mn, off);
                        umma_commit_cg<CG>(bar(info.empty[rp.slot]));
                    }
                    __syncwarp();
                }
                if (elect_one()) umma_commit_cg<CG>(bar(info.accf[buf]));
                __syncwarp();
            }
        }
        __syncwarp();
    } else if (warp < EW0) {
        // ============================================================ gathers
        // Stage g (counted over the CTA's units) belongs to warp g % GWN.  The
        // first CTA's warps arrive on the stage's barrier, the second one's
        // add BULK_SIGNAL_BYTES to the bytes that it waits for.
        const int w = warp - GW0;
        RingPos rp;                 // the warp's next stage
        rp.advance(w, nst);
        uint32_t mine = w;          // stages until the warp's next one
        bool wrapped = false, v_ready = false;
        auto begin = [&]() {        // the stage's slot is free
            if (wrapped) wait_bar(info.empty[rp.slot], rp.phase ^ 1u);
            ok = __all_sync(0xffffffffu, ok);
        };
        auto next_stage = [&]() {
            const uint32_t before = rp.slot;
            rp.advance(GWN, nst);
            wrapped = wrapped || rp.slot <= before;
            mine += GWN;
        };
        auto finish = [&]() {       // the warp's copies have landed; on to its next stage
            cp_async_commit();
            cp_async_wait<0>();
            fence_async_smem();
            __syncwarp();
            if (lane == 0) {
                if (rank == 0) mbar_arrive_release(bar(info.full[rp.slot]));
                else bulk_signal_leader(smem_u32(info.token), bar(info.full[rp.slot]));
            }
            next_stage();
        };
        uint32_t xoff[BM / 4];      // this lane's token rows (row 4 i + lane / 8), in 16-byte units of x
        int mt_of = -1, rows = 0;
        const uint32_t d16 = (uint32_t)p.d_in >> 3;
        for (int u = cl; u < n_units && ok; u += n_cl) {
            const int tile = u / KS, s = u - tile * KS, mt = tile % n_mt, n0 = tile / n_mt * BN + rank * NB;
            const int m0 = (mt * CG + rank) * BM;
            const bool lin = !(info.mt_x0[mt] & X_GATHER);
            if (mt != mt_of && !lin) {
                mt_of = mt;
                rows = max(0, min(BM, T - m0));
#pragma unroll
                for (int i = 0; i < BM / 4; ++i) {
                    const int r = 4 * i + (lane >> 3);
                    xoff[i] = r < rows ? (uint32_t)p.perm[m0 + r] : 0u;
                }
#pragma unroll
                for (int i = 0; i < BM / 4; ++i) xoff[i] = xoff[i] * d16 + (uint32_t)(lane & 7);
            }
            const int k0 = chunk_lo(s), n = chunk_lo(s + 1) - k0;
            const uint32_t sw = (uint32_t)swz128(lane >> 3, lane & 7);  // row 4 i + lane / 8: swizzle by (4 i + lane / 8) % 8
            while ((int)mine < n && ok) {
                begin();
                if (!ok) break;
                if (lin) {  // the TMA warp loads the rows
                    if (lane == 0 && rank == 0) mbar_arrive_relaxed(bar(info.full[rp.slot]));
                    next_stage();
                    continue;
                }
                const int kc = k0 + (int)mine;
                const uint32_t xs = ring32 + rp.slot * stage;
                const bool in = kc * BK + (lane & 7) * 8 < p.d_in;
                const uint16_t *xk = p.x + (in ? (int64_t)kc * BK : 0);
#pragma unroll
                for (int i = 0; i < BM / 4; ++i)
                    if (4 * i + (lane >> 3) < rows)
                        cp_async16(xs + ((sw + i * 512) ^ ((i & 1) << 6)), xk + (uint64_t)xoff[i] * 8, in);
                finish();
            }
            mine -= n;
            // delta chunk j of the tile belongs to split j % KS
            const int b1 = info.mt_b1[mt];
            int j = 0;
            if (n_delta(mt, s) > 0 && !v_ready) {
                pdl_wait();  // the V tiles are the shrink's
                v_ready = true;
            }
            for (int bb = info.mt_b0[mt]; bb < b1 && ok; bb += 32) {
                // 32 blocks at a time: lane l holds block bb + l
                int4 r0 = make_int4(0, 0, -1, 0);
                int S = 0;
                if (bb + lane < b1) {
                    r0 = *reinterpret_cast<const int4 *>(p.blk + BLK_INTS * (bb + lane));
                    S = r0.w + p.blk[BLK_INTS * (bb + lane) + BLK_NRES];
                    if (S > S_MAX || S <= 0 || r0.y <= 0) S = 0;
                }
                const int nb = min(32, b1 - bb);
                for (int i = 0; i < nb && ok; ++i) {
                    const int Sb = __shfl_sync(0xffffffffu, S, i);
                    for (int c0 = 0; c0 < Sb; c0 += BK, ++j) {
                        if (j % KS != s) continue;
                        if (mine > 0) {
                            --mine;
                            continue;
                        }
                        const int start = __shfl_sync(0xffffffffu, r0.x, i), M = __shfl_sync(0xffffffffu, r0.y, i);
                        const int d = __shfl_sync(0xffffffffu, r0.z, i), rc = __shfl_sync(0xffffffffu, r0.w, i);
                        const int b = bb + i, kn = min(BK, ((Sb + 15) & ~15) - c0);  // stack rows, padded to 16
                        // the lane's two stacked B rows
                        const uint16_t *src[2];
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int k = c0 + h * 32 + lane;
                            src[h] = k >= Sb ? nullptr
                                     : k < rc ? p.B + ((int64_t)d * p.rc_max + k) * p.d_out
                                              : res_b_row(p, p.blk_res[(int64_t)b * S_MAX + (k - rc)]);
                        }
                        begin();
                        if (!ok) break;
                        const uint32_t xs = ring32 + rp.slot * stage, ws = xs + x_bytes;
                        // V rows of the block at their tile rows (other rows zero)
                        const uint16_t *vt = p.vext + (int64_t)b * (TM * VEXT_COLS) + c0;
                        for (int idx = lane; idx < m_rows * 8; idx += 32) {
                            const int r = idx >> 3, c = idx & 7, iv = m0 + r - start;
                            const bool in = iv >= 0 && iv < M && c * 8 < kn;
                            cp_async16(xs + swz128(r, c), vt + (in ? iv * VEXT_COLS + c * 8 : 0), in);
                        }
                        // stacked B rows, this CTA's columns, as 64-wide MN-major parts;
                        // 8 or 16 pieces of 16 bytes a row (kn times that is a
                        // multiple of 32: every lane takes part in every round)
                        const int lg = NB == 128 ? 4 : 3;
                        for (int idx = lane; idx < kn << lg; idx += 32) {
                            const int k = idx >> lg, c = idx & ((1 << lg) - 1), col = n0 + c * 8;
                            const uint64_t lo = (uint64_t)__shfl_sync(0xffffffffu, (unsigned long long)src[0], k & 31);
                            const uint64_t hi = (uint64_t)__shfl_sync(0xffffffffu, (unsigned long long)src[1], k & 31);
                            const uint16_t *sp = reinterpret_cast<const uint16_t *>(k < 32 ? lo : hi);
                            const bool in = sp != nullptr && col < p.d_out;
                            cp_async16(ws + (c >> 3) * 8192 + swz128(k, c & 7), in ? sp + col : p.x, in);
                        }
                        if (lane == 0) {
                            const int r0 = start - mt * (BM * CG);  // the block's first row in the tile
                            info.dstage[rp.slot] = (uint32_t)(kn >> 4) | (uint32_t)max(r0, 0) << 10 |
                                                   (uint32_t)min(r0 + M, BM * CG) << 20;
                        }
                        finish();
                        mine -= 1;  // this stage itself
                    }
                }
            }
        }
    } else {
        // ============================================================ epilogue
        const int q = warp & 3, row = q * 32 + lane, et = tid - 32 * EW0;
        const bool wide = (p.d_out & 15) == 0 && (reinterpret_cast<uintptr_t>(p.y) & 31) == 0;
        uint32_t lt = 0;
        const bool share = n_units <= n_cl;  // one unit a CTA
        if (KS > 1) pdl_wait();  // the partials' workspace is the shrink's
        for (int u = cl; u < n_units; u += n_cl, ++lt) {
            const int tile = u / KS, mt = tile % n_mt, n0 = tile / n_mt * BN;
            const uint32_t buf = lt & 1;
            const int m0 = (mt * CG + rank) * BM, gp = m0 + row;
            const int tok = gp < T ? p.perm[gp] : -1;
            wait_bar(info.accf[buf], (lt >> 1) & 1);
            tc_fence_after();
            const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + buf * BN;
            const int rows = max(0, min(BM, T - m0));
            float *part = p.part + ((int64_t)u * CG + rank) * (m_rows * BN);
            uint16_t *yr = p.y + (int64_t)max(tok, 0) * p.d_out;
            if (q * 32 < rows) {
#pragma unroll 1
                for (int c = 0; c < BN; c += 32) {
                    uint32_t v[2][16];
                    tmem_ld16(ta + c, v[0]);
                    tmem_ld16(ta + c + 16, v[1]);
                    tmem_ld_wait();
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int col = n0 + c + 16 * h;
                        if (tok < 0) continue;
                        if (KS > 1) {  // [8 columns][row][8]: a warp's stores are contiguous
#pragma unroll
                            for (int i = 0; i < 2; ++i)
                                store_part8(part + ((c >> 3) + 2 * h + i) * (m_rows * 8) + row * 8, v[h] + 8 * i);
                            continue;
                        }
                        uint32_t w[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            w[i] = pack_bf16(__uint_as_float(v[h][2 * i]), __uint_as_float(v[h][2 * i + 1]));
                        if (col + 8 < p.d_out) store32(yr + col, w, wide);
                        else if (col < p.d_out) *reinterpret_cast<uint4 *>(yr + col) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_relaxed_cluster<CG>(leader_addr<CG>(bar(info.acce[buf])));
            if (KS == 1) continue;
            // Sum the partials of the tile (this CTA's rows) in split order, a
            // share of them per split.  ctr[0] counts the splits stored (low
            // half) and marks the ones that left their share to the split
            // that stores last (high half).  Where every unit may run at once
            // a split waits a while for the others (about 0.1 ms) and then
            // leaves; so nothing depends on the CTAs of a tile running
            // together, which other streams' launches can prevent.  (Leaving
            // at once: an 8B layer at 24 tokens 195 us, 175 with the wait.)
            __threadfence();
            named_sync(BAR_E, EPI_N);
            uint32_t *ctr = p.ctr + 2 * (tile * CG + rank);
            if (et == 0) {
                const uint32_t own = 1u << (u - tile * KS);
                uint32_t c = atomicAdd(ctr, 1u), sum = own;
                if ((c & 0xffffu) + 1u == (uint32_t)KS) {
                    sum |= c >> 16;
                } else {
                    bool all = false;
                    for (int i = 0; i < SPLIT_POLLS && share && !all; ++i) {
                        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(c) : "l"(ctr) : "memory");
                        all = (c & 0xffffu) == (uint32_t)KS;
                        if (!all) __nanosleep(32);
                    }
                    if (!all && (atomicOr(ctr, own << 16) & 0xffffu) != (uint32_t)KS) sum = 0u;
                }
                info.shares = sum;
                __threadfence();
            }
            named_sync(BAR_E, EPI_N);
            const uint32_t shares = info.shares;
            if (!shares) continue;
            const float *p0 = p.part + ((int64_t)tile * KS * CG + rank) * (m_rows * BN);
            const int64_t ps = (int64_t)CG * m_rows * BN;
            const int lc = BN == 256 ? 5 : 4, n_all = rows << lc;
            // consecutive shares together
            for (uint32_t left = shares; left;) {
                const int s0 = __ffs(left) - 1, n = __ffs(~(left >> s0)) - 1, n_it = n_all * (s0 + n) / KS;
                left &= ~(((1u << n) - 1u) << s0);
                // (row, 8 columns) items, two a round per thread, up to four splits' loads in flight
                for (int base = n_all * s0 / KS + et; base < n_it; base += 2 * EPI_N) {
                    float a[2][8] = {};
                    for (int k0 = 0; k0 < KS; k0 += 4) {
                        float4 v[2][4][2];
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int s = 0; s < 4; ++s) {
                                const int it = base + h * EPI_N;
                                if (it < n_it && k0 + s < KS) {
                                    const int c8 = it & ((1 << lc) - 1), r = it >> lc;
                                    const float4 *src = reinterpret_cast<const float4 *>(p0 + (k0 + s) * ps + (c8 * m_rows + r) * 8);
                                    v[h][s][0] = __ldcg(src);
                                    v[h][s][1] = __ldcg(src + 1);
                                } else {
                                    v[h][s][0] = v[h][s][1] = make_float4(0.f, 0.f, 0.f, 0.f);
                                }
                            }
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int s = 0; s < 4; ++s) {
                                a[h][0] += v[h][s][0].x;
                                a[h][1] += v[h][s][0].y;
                                a[h][2] += v[h][s][0].z;
                                a[h][3] += v[h][s][0].w;
                                a[h][4] += v[h][s][1].x;
                                a[h][5] += v[h][s][1].y;
                                a[h][6] += v[h][s][1].z;
                                a[h][7] += v[h][s][1].w;
                            }
                    }
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int it = base + h * EPI_N;
                        if (it >= n_it) continue;
                        const int r = it >> lc, col = n0 + (it & ((1 << lc) - 1)) * 8;
                        if (col < p.d_out)
                            *reinterpret_cast<uint4 *>(p.y + (int64_t)p.perm[m0 + r] * p.d_out + col) =
                                make_uint4(pack_bf16(a[h][0], a[h][1]), pack_bf16(a[h][2], a[h][3]),
                                           pack_bf16(a[h][4], a[h][5]), pack_bf16(a[h][6], a[h][7]));
                    }
                }
            }
            // every share summed: zero for the next launch
            if (et == 0) {
                const uint32_t n = __popc(shares);
                if (atomicAdd(ctr + 1, n) + n == (uint32_t)KS) {
                    atomicExch(ctr, 0u);
                    atomicExch(ctr + 1, 0u);
                }
            }
        }
    }
    pdl_wait();  // the launch completes after the shrink has
    if (!ok) {
        atomicOr(p.err, SALT_DEVERR_TIMEOUT);
        __nanosleep(1000000);  // copies already issued land before the CTA may exit
    }
    __syncwarp();
    tc_fence_before();
    cta_or_cluster_sync<CG>();
    if (warp == 1) tmem_dealloc<CG>(tmem, 2 * BN);
}

int g_base_sms[64];    // SMs per device, and the CTA pairs that fit on them at once (filled by base_prepare)
int g_base_pairs[64];

struct BasePlan {
    int cg, bn, ks, shrink_ctas;
};

// The launch's shape, by an estimate of its time in us: the tile width, the K
// splits, and the SMs the shrink gets.  Either the shrink takes every SM and
// the K loop starts after it, or it takes 24 or 48 beside the K loop on the
// others (only the delta waits for it): worth it where the K loop is long or
// leaves SMs idle anyway, e.g. 24 tokens of 4096 x 14336 45 -> 36 us beside,
// but 14336 x 4096 at 512 tokens 75 us in turn against 89.
// The constants are fits to measured launches of 24 to 1024 tokens, d_in 4096
// and 14336, d_out 1024 to 14336; the estimate only ranks shapes, and its steps
// (the tail at 8 tiles of tokens, no shrink beside above 2048 tokens) are rough.
// Outside the fits, measured: 129, 200 and 300 tokens of 1024 x 1024 14.7, 14.9
// and 15.2 us, of 4096 x 1024 24.4, 23.5 and 23.9; 2048 and 2049 tokens of
// 4096 x 4096 62.9 and 62.9, of 8192 x 3072 86 and 113 (one wave more).  A shrink
// beside above 2048 tokens gives as much as it takes: us in turn / beside at
// 2560 tokens of 4096 x 1024 39.8 / 32.4, of 2048 x 2048 32.8 / 35.8, at 8192 of
// 8192 x 3072 293 / 278, of 14336 x 512 150 / 158.
BasePlan base_plan(int T, int d_in, int d_out, int n_blk, int n_sm, int max_pairs)
{
    const int nk = (d_in + BK - 1) / BK, cg = T > BM ? 2 : 1;
    const int n_mt = (T + BM * cg - 1) / (BM * cg), m_rows = cg == 2 ? BM : (std::min(T, BM) + 15) & ~15;
    BasePlan best = {cg, 128, 1, 0};
    double best_t = 1e30;
    for (int beside = 0; beside <= 48; beside += 24) {
        if (beside && (T > 2048 || n_sm < 2 * beside)) break;
        const int sms = n_sm - beside, n_cl = std::max(1, cg == 2 ? std::min(max_pairs, sms / 2) : sms);
        const int sh = beside ? beside : n_sm, sh_ks = std::max(1, std::min(16, sh / std::max(1, n_blk)));
        const int sh_waves = (n_blk * sh_ks + sh - 1) / sh;
        const double t_shrink = 12.0 + 0.42 * sh_waves * ((nk + sh_ks - 1) / sh_ks);
        for (int bn = 128; bn <= (cg == 2 ? 256 : 128); bn *= 2) {
            const int64_t tiles = (int64_t)n_mt * ((d_out + bn - 1) / bn);
            for (int ks = 1; ks <= std::min(BASE_KS_MAX, nk); ++ks) {
                const int64_t units = tiles * ks;
                if (ks > 1 && (units * cg * m_rows * bn > (int64_t)PART_CAP * TM * PART_COLS || 2 * tiles * cg > BASE_CTRS)) break;
                const double waves = (double)((units + n_cl - 1) / n_cl);
                // a chunk: one CTA a tile is bound by streaming W from memory
                // (16 KB a chunk at 6 TB/s over the running CTAs, or by its
                // own latency), a pair by its stages
                const double active = (double)std::min<int64_t>(units, n_cl);
                const double chunk = cg == 1 ? std::max(0.36, 0.41 * active / n_sm) : (bn == 256 ? 0.35 : 0.23);
                const double k_loop = ((nk + ks - 1) / ks) * chunk, tail = n_mt > 8 ? 1.0 : cg == 2 ? 9.0 : 4.0;
                const bool share = units <= n_cl;
                const double split = ks == 1 ? 0 : (m_rows / 128.0) * (bn / 128.0) * (share ? 2.0 : 0.5 + 0.8 * ks) + 2.0;
                const double gemm = waves * (k_loop + tail) + split;
                // (a K loop that follows the shrink still overlaps its tail)
                const double t = beside ? gemm + std::max(0.0, t_shrink - k_loop) : gemm + t_shrink - std::min(3.0, k_loop);
                if (t < best_t) {
                    best_t = t;
                    best = {cg, bn, ks, beside};
                }
            }
        }
    }
    return best;
}

// The plan of a launch on the current device; false when it is not prepared.
bool plan_here(int T, int d_in, int d_out, int n_blk, BasePlan *pl, int *n_cl)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || g_base_sms[dev] <= 0) return false;
    *pl = base_plan(T, d_in, d_out, n_blk, g_base_sms[dev], g_base_pairs[dev]);
    const int sms = g_base_sms[dev] - pl->shrink_ctas;
    *n_cl = std::max(1, pl->cg == 2 ? std::min(g_base_pairs[dev], sms / 2) : sms);
    return true;
}

}  // namespace

cudaError_t base_prepare(int device)
{
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    cudaError_t e = cudaDeviceGetAttribute(&g_base_sms[device], cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(salt_base_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BASE_SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(salt_base_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)BASE_SMEM);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((g_base_sms[device] & ~1) > 0 ? g_base_sms[device] & ~1 : 2, 1, 1);
    cfg.blockDim = dim3(BASE_THREADS, 1, 1);
    cfg.dynamicSmemBytes = BASE_SMEM;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(&g_base_pairs[device], salt_base_kernel<2>, &cfg);
}

int base_shrink_ctas(int T, int d_in, int d_out, int n_blk)
{
    BasePlan pl;
    int n_cl;
    return plan_here(T, d_in, d_out, n_blk, &pl, &n_cl) ? pl.shrink_ctas : 0;
}

bool base_launch_shape(int T, int d_in, int d_out, int n_blk, salt_base_shape *out)
{
    BasePlan pl;
    int max_cl;
    if (!plan_here(T, d_in, d_out, n_blk, &pl, &max_cl)) return false;
    const int bm = BM * pl.cg;
    out->cta_group = pl.cg;
    out->tile_cols = pl.bn;
    out->k_splits = pl.ks;
    out->shrink_ctas = pl.shrink_ctas;
    out->units = ((T + bm - 1) / bm) * ((d_out + pl.bn - 1) / pl.bn) * pl.ks;
    out->clusters = std::min(out->units, max_cl);
    return true;
}

cudaError_t launch_base(BaseParams &p, const uint16_t *W, int n_blk, cudaStream_t stream)
{
    BasePlan pl;
    int max_cl;
    if (!plan_here(p.T, p.d_in, p.d_out, n_blk, &pl, &max_cl)) return cudaErrorInvalidDevice;
    cudaError_t e;
    p.bn = pl.bn;
    p.ks = pl.ks;
    const cuuint32_t nb = (cuuint32_t)(pl.bn / pl.cg);
    // W_base[d_in][d_out]: boxes of 64 K rows x 64 N columns;
    // W_base[d_out][d_in]: NB rows x 64 K
    e = p.w_layout == SALT_W_IN_OUT ? encode_map_2d(&p.wmap, W, p.d_out, p.d_in, 64, 64)
                                    : encode_map_2d(&p.wmap, W, p.d_in, p.d_out, 64, nb);
    if (e == cudaSuccess) e = encode_map_2d(&p.xmap, p.x, p.d_in, p.T, 64, BM);
    if (e != cudaSuccess) return e;
    const int bm = BM * pl.cg;
    const int64_t units = (int64_t)((p.T + bm - 1) / bm) * ((p.d_out + pl.bn - 1) / pl.bn) * pl.ks;
    const int n_cl = (int)std::min<int64_t>(units, max_cl);
    if (n_cl <= 0) return cudaSuccess;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = pl.cg;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.gridDim = dim3(n_cl * pl.cg, 1, 1);
    cfg.blockDim = dim3(BASE_THREADS, 1, 1);
    cfg.dynamicSmemBytes = BASE_SMEM;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return pl.cg == 2 ? cudaLaunchKernelEx(&cfg, salt_base_kernel<2>, p) : cudaLaunchKernelEx(&cfg, salt_base_kernel<1>, p);
}

}  // namespace salt
