// Segment builder: groups a heterogeneous batch for the apply kernel.
//
// Section "Multi-Tenant Serving" groups requests by their (centroid, gamma)
// pair, and the residuals are batched heterogeneously (SGMV, Section
// "Multi-Tenant LoRA Serving").  One CTA of 1024 threads:
//   1. validates every (domain, gamma bin, slot) id into the device error
//      word (an invalid id is treated as -1, never dereferenced; a token
//      without a centroid has no bin),
//   2. sorts the keys (domain + 1, bin + 1, slot + 1, token): up to 1024 by a
//      bitonic network, one key a thread; more by a stable LSD radix sort in
//      shared memory, over only the bits that the context's domain, bin and
//      slot counts need (two passes of 7 for 640 slots and 8 domains).
//      Tokens enter in token order, so ties stay in it,
//   3. writes perm / sorted_slot and the maximal (domain, bin) and user runs
//      (run heads counted by ballots, one scan over the warps),
//   4. cuts row blocks for the apply kernel: within a domain (over all of
//      its bins), user runs are grouped umax at a time and each group is
//      split evenly into ceil(len / TM) blocks of at most TM tokens.  gamma
//      enters as each token's centroid scale s_c(domain) * gamma[bin], so the
//      bins of one centroid share its blocks and factor reads.  The leading
//      (-1, -1) run (tokens with neither term) gets no block, so those rows
//      are never touched.
//
// One CTA is bound by its chains of dependent loads and barriers, not by
// bytes: token order is kept warp by warp (warp w holds 32 * R consecutive
// positions), so table writes are coalesced, and the loads of four rounds are
// in flight together.
// Measured (16384 tokens with gamma bins, 48 users): 519 -> 85 us a build
// against two bitonic networks through shared memory and per-thread chunks
// of positions; 512 tokens of 640 slots take 22.6 us as before.
#include "salt_internal.cuh"

namespace salt {
namespace {

// A key: token | slot + 1 | gamma bin + 1 | domain + 1 from the low bits up
// (the grouped order), or with the slot above the bin (the apply order); the
// fields above the token are as wide as the context's counts need.
constexpr int KEY_TOK_BITS = 14;
static_assert(SALT_MAX_TOKENS <= (1 << KEY_TOK_BITS), "a token index must fit the key");
constexpr int RADIX_BITS = 8;
constexpr int SEG_WARPS = SEG_THREADS / 32;
constexpr int MAX_ROUNDS = (SALT_MAX_TOKENS + SEG_THREADS - 1) / SEG_THREADS;  // 32-token rounds a warp holds
constexpr int LOAD_BATCH = 4;                                                  // rounds whose loads are in flight together

struct KeyLayout {
    int slot_bits, gb_bits, dom_bits;
    bool slot_high;  // apply order: slot above the bin
    __device__ int slot_at() const { return KEY_TOK_BITS + (slot_high ? gb_bits : 0); }
    __device__ int gb_at() const { return KEY_TOK_BITS + (slot_high ? 0 : slot_bits); }
    __device__ int dom_at() const { return KEY_TOK_BITS + slot_bits + gb_bits; }
    __device__ uint64_t make(int d, int gb, int s, int t) const
    {
        return (uint64_t)(d + 1) << dom_at() | (uint64_t)(gb + 1) << gb_at() | (uint64_t)(s + 1) << slot_at() | (uint64_t)t;
    }
    __device__ int dom(uint64_t k) const { return (int)(k >> dom_at()) - 1; }
    __device__ int gb(uint64_t k) const { return (int)((k >> gb_at()) & ((1u << gb_bits) - 1)) - 1; }
    __device__ int slot(uint64_t k) const { return (int)((k >> slot_at()) & ((1u << slot_bits) - 1)) - 1; }
    __device__ static int tok(uint64_t k) { return (int)(k & ((1u << KEY_TOK_BITS) - 1)); }
    // equal for tokens of one run: the grouped order's (domain, bin) or the
    // apply order's domain; and the user runs below it
    __device__ uint64_t cent(uint64_t k) const { return slot_high ? k >> dom_at() : k >> gb_at(); }
    __device__ uint64_t user(uint64_t k) const { return slot_high ? k >> slot_at() : k >> KEY_TOK_BITS; }
};
__device__ __forceinline__ int bits_for(int n) { return n > 1 ? 32 - __clz(n - 1) : 0; }  // values 0 .. n - 1

// Exclusive scan of one int per thread over the whole block; *total gets the sum.
__device__ int block_exclusive_scan(int v, int *total, int *warp_sums)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < nwarps ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        warp_sums[lane] = w;  // inclusive
    }
    __syncthreads();
    int before = (warp ? warp_sums[warp - 1] : 0) + x - v;
    *total = warp_sums[nwarps - 1];
    __syncthreads();
    return before;
}

// One stable pass: the n keys reordered by the digit at `shift` of `bits`
// (<= RADIX_BITS).  Whole block; warp w holds positions [32 R w, 32 R (w + 1)).
// hist is [warps that hold positions][1 << bits].
__device__ void radix_pass(uint64_t *keys, uint32_t *hist, int n, int R, int shift, int bits, int *warp_sums)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nd = 1 << bits;
    const uint32_t dmask = (uint32_t)nd - 1u;
    const int nw = (n + 32 * R - 1) / (32 * R);
    for (int i = tid; i < nw * nd; i += SEG_THREADS) hist[i] = 0;
    uint64_t k[MAX_ROUNDS];
    uint32_t rank[MAX_ROUNDS / 2];  // rank among the warp's equal digits, two to a word
    __syncthreads();
    uint32_t *h = hist + warp * nd;
#pragma unroll
    for (int i = 0; i < MAX_ROUNDS; ++i) {
        if (i >= R) break;
        const int pos = (warp * R + i) * 32 + lane;
        const unsigned act = __ballot_sync(0xffffffffu, pos < n);
        uint32_t r = 0;
        if (pos < n) {
            k[i] = keys[pos];
            const uint32_t d = (uint32_t)(k[i] >> shift) & dmask;
            const unsigned m = __match_any_sync(act, d);
            const int below = __popc(m & ((1u << lane) - 1u));
            r = h[d] + below;
            __syncwarp(act);
            if (below == 0) h[d] += __popc(m);
            __syncwarp(act);
        }
        rank[i / 2] = (i & 1) ? rank[i / 2] | r << 16 : r;
    }
    __syncthreads();
    // exclusive prefix over (digit, warp)
    uint32_t sum = 0;
    if (tid < nd) {
#pragma unroll 8
        for (int w = 0; w < nw; ++w) sum += hist[w * nd + tid];
    }
    int total;
    uint32_t run = (uint32_t)block_exclusive_scan((int)sum, &total, warp_sums);
    if (tid < nd)
#pragma unroll 8
        for (int w = 0; w < nw; ++w) {
            const uint32_t c = hist[w * nd + tid];
            hist[w * nd + tid] = run;
            run += c;
        }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < MAX_ROUNDS; ++i) {
        if (i >= R) break;
        if ((warp * R + i) * 32 + lane < n) {
            const uint32_t d = (uint32_t)(k[i] >> shift) & dmask;
            keys[h[d] + ((rank[i / 2] >> (16 * (i & 1))) & 0xffffu)] = k[i];
        }
    }
    __syncthreads();
}

// Ascending bitonic sort of n <= SEG_THREADS distinct keys, one a thread:
// strides below 32 by shuffles, only the longer ones (10 of 45 at 512 keys)
// through shared memory.
__device__ void bitonic_sort(uint64_t *keys, int n)
{
    const int tid = threadIdx.x;
    uint64_t v = tid < n ? keys[tid] : ~0ull;
    int n2 = 32;
    while (n2 < n) n2 <<= 1;
    for (int k = 2; k <= n2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
            uint64_t o;
            if (j >= 32) {
                __syncthreads();
                if (tid < n2) keys[tid] = v;  // (past the keys: the histogram's region, unused here)
                __syncthreads();
                o = tid < n2 ? keys[tid ^ j] : v;
            } else {
                o = __shfl_xor_sync(0xffffffffu, v, j);
            }
            const bool keep_min = ((tid & j) == 0) == ((tid & k) == 0);
            v = keep_min == (v < o) ? v : o;
        }
    __syncthreads();
    if (tid < n) keys[tid] = v;
    __syncthreads();
}

// Sort of n distinct keys that lie in token order, by the bits [lo, hi)
// and then by what lies below in their present order: the radix passes
// (even, <= RADIX_BITS) are stable; a batch of one key a thread is sorted by
// whole keys, which their low bits (bin and token) put in the same order.
__device__ void radix_sort(uint64_t *keys, uint32_t *hist, int n, int R, int lo, int hi, int *warp_sums)
{
    if (n <= SEG_THREADS) {  // 512 keys: 22.1 us a build, 23.4 by two radix passes
        bitonic_sort(keys, n);
        return;
    }
    const int passes = (hi - lo + RADIX_BITS - 1) / RADIX_BITS;
    for (int i = 0; i < passes; ++i) {
        const int a = lo + (hi - lo) * i / passes, b = lo + (hi - lo) * (i + 1) / passes;
        radix_pass(keys, hist, n, R, a, b - a, warp_sums);
    }
}

__global__ void __launch_bounds__(SEG_THREADS, 1) seg_build_kernel(SegParams p)
{
    extern __shared__ __align__(16) uint64_t keys[];
    __shared__ int warp_sums[32];
    __shared__ int max_stack;
    const int T = p.T;
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5;

    if (T == 0) {
        if (tid == 0) {
            p.s.dseg_ptr[0] = 0;
            p.s.useg_ptr[0] = 0;
            p.s.counts[0] = p.s.counts[1] = p.s.counts[2] = p.s.counts[3] = p.s.counts[4] = 0;
        }
        return;
    }
    const int R = (T + SEG_THREADS - 1) / SEG_THREADS;
    uint32_t *hist = reinterpret_cast<uint32_t *>(keys + T);
    KeyLayout L;
    L.slot_bits = bits_for(p.n_slots + 1);
    L.gb_bits = p.has_gbin ? bits_for(p.n_gamma + 1) : 0;
    L.dom_bits = bits_for(p.n_domains + 1);
    L.slot_high = false;

    // 1. validate and build keys
    uint32_t errbits = 0;
    const int32_t *dom_ids = p.dom_ids, *slot_ids = p.slot_ids, *gb_ids = p.gb_ids;
    for (int i0 = 0; i0 < R; i0 += LOAD_BATCH) {
        int d[LOAD_BATCH], sl[LOAD_BATCH], gb[LOAD_BATCH], rc[LOAD_BATCH], rk[LOAD_BATCH];
        uint64_t magic[LOAD_BATCH];
#pragma unroll
        for (int i = 0; i < LOAD_BATCH; ++i) {
            const int pos = (warp * R + i0 + i) * 32 + lane;
            const bool in = i0 + i < R && pos < T;
            d[i] = in ? dom_ids[pos] : -1;
            sl[i] = in ? slot_ids[pos] : -1;
            gb[i] = in && p.has_gbin ? gb_ids[pos] : -1;
        }
#pragma unroll
        for (int i = 0; i < LOAD_BATCH; ++i) {
            rc[i] = d[i] >= 0 && d[i] < p.n_domains ? p.dom_rc[d[i]] : 0;
            magic[i] = 0;
            rk[i] = 0;
            if (sl[i] >= 0 && sl[i] < p.n_slots) {
                const uint8_t *h = p.pool + (int64_t)sl[i] * p.slot_stride;
                magic[i] = *reinterpret_cast<const uint64_t *>(h);
                rk[i] = *reinterpret_cast<const int32_t *>(h + 12);
            }
        }
#pragma unroll
        for (int i = 0; i < LOAD_BATCH; ++i) {
            const int pos = (warp * R + i0 + i) * 32 + lane;
            if (i0 + i >= R || pos >= T) continue;
            int dd = d[i], s = sl[i], g = -1;
            if (dd < -1 || dd >= p.n_domains) {
                errbits |= SALT_DEVERR_DOMAIN_RANGE;
                dd = -1;
            } else if (dd >= 0 && rc[i] <= 0) {
                errbits |= SALT_DEVERR_DOMAIN_NOT_PINNED;
                dd = -1;
            }
            if (p.has_gbin && dd >= 0) {
                g = gb[i];
                if (g < -1 || g >= p.n_gamma) {
                    errbits |= SALT_DEVERR_GAMMA_RANGE;
                    g = -1;
                }
            }
            if (s < -1 || s >= p.n_slots) {
                errbits |= SALT_DEVERR_SLOT_RANGE;
                s = -1;
            } else if (s >= 0) {
                if (magic[i] != SALT_BLOB_MAGIC) {
                    errbits |= SALT_DEVERR_SLOT_EMPTY;
                    s = -1;
                } else if (rk[i] < 1 || rk[i] > p.r_max) {
                    errbits |= SALT_DEVERR_RANK;
                    s = -1;
                }
            }
            keys[pos] = L.make(dd, g, s, pos);
        }
    }
    if (errbits) atomicOr(p.err, errbits);
    __syncthreads();

    // 2. the grouped order
    radix_sort(keys, hist, T, R, KEY_TOK_BITS, L.dom_at() + L.dom_bits, warp_sums);
    const bool skip0 = L.dom(keys[0]) == -1 && L.slot(keys[0]) == -1;

    // Run heads of the keys in the order L, by ballot: counted, scanned over
    // the warps, then f(pos, key, domain head, user head, runs before this
    // position) for every position.  A position's own run is the count of
    // heads up to it, less one.
    auto for_runs = [&](int &n_d, int &n_u, auto f) {
        int nd = 0, nu = 0;
        for (int i = 0; i < R; ++i) {
            const int pos = (warp * R + i) * 32 + lane;
            bool dh = false, uh = false;
            if (pos < T) {
                const uint64_t k = keys[pos];
                const uint64_t kp = pos ? keys[pos - 1] : ~k;
                dh = pos == 0 || L.cent(k) != L.cent(kp);
                uh = pos == 0 || L.user(k) != L.user(kp);
            }
            nd += __popc(__ballot_sync(0xffffffffu, dh));
            nu += __popc(__ballot_sync(0xffffffffu, uh));
        }
        // (each warp counts once, in its lane 0)
        int od = block_exclusive_scan(lane == 0 ? nd : 0, &n_d, warp_sums);
        int ou = block_exclusive_scan(lane == 0 ? nu : 0, &n_u, warp_sums);
        od = __shfl_sync(0xffffffffu, od, 0);
        ou = __shfl_sync(0xffffffffu, ou, 0);
        const unsigned lt = (1u << lane) - 1u;
        for (int i = 0; i < R; ++i) {
            const int pos = (warp * R + i) * 32 + lane;
            bool dh = false, uh = false;
            uint64_t k = 0;
            if (pos < T) {
                k = keys[pos];
                const uint64_t kp = pos ? keys[pos - 1] : ~k;
                dh = pos == 0 || L.cent(k) != L.cent(kp);
                uh = pos == 0 || L.user(k) != L.user(kp);
            }
            const unsigned md = __ballot_sync(0xffffffffu, dh), mu = __ballot_sync(0xffffffffu, uh);
            if (pos < T) f(pos, k, dh, uh, od + __popc(md & lt), ou + __popc(mu & lt));
            od += __popc(md);
            ou += __popc(mu);
        }
    };
    auto token_scale = [&](int d, int gb) {
        return d >= 0 ? p.dom_sc[d] * (gb >= 0 ? p.gamma[gb] : 1.f) : 0.f;
    };

    // 3. the grouped order's tables and runs; without gamma bins it is the
    //    apply order too
    int n_dseg, n_useg;
    for_runs(n_dseg, n_useg, [&](int i, uint64_t k, bool dh, bool uh, int od, int ou) {
        const int d = L.dom(k), gb = p.has_gbin ? L.gb(k) : -1, s = L.slot(k);
        p.s.perm[i] = L.tok(k);
        if (dh) {
            p.s.dseg_ptr[od] = i;
            p.s.dseg_dom[od] = d;
            p.s.dseg_gbin[od] = gb;
        }
        if (uh) {
            p.s.useg_ptr[ou] = i;
            p.s.useg_dom[ou] = d;
            p.s.useg_gbin[ou] = gb;
            p.s.useg_slot[ou] = s;
        }
        if (!p.has_gbin) {
            p.s.aperm[i] = L.tok(k);
            p.s.sorted_slot[i] = s;
            p.s.tok_sc[i] = token_scale(d, -1);
            if (dh) p.s.d_first[od] = ou;
            if (uh) p.s.u_drun[ou] = od + (dh ? 1 : 0) - 1;
        }
    });
    if (tid == 0) {
        p.s.dseg_ptr[n_dseg] = T;
        p.s.useg_ptr[n_useg] = T;
    }
    // The runs the row blocks are cut from: the grouped order's, unless the
    // batch has gamma bins (below).
    const int32_t *uptr = p.s.useg_ptr, *udom = p.s.useg_dom;
    int n_ur = n_useg;
    if (p.has_gbin) {
        // 3'. The apply order: the keys stably sorted by (domain, slot), so
        //     that a user's tokens in several bins form one run and take one
        //     set of residual rows in a block (gamma is applied per token);
        //     within a run the grouped order's (bin, token) stays.  Writes
        //     aperm and, in this order, sorted_slot, tok_sc and the domain
        //     and (domain, slot) runs.
        __syncthreads();  // every thread is done with the grouped order
        KeyLayout A = L;
        A.slot_high = true;
        for (int i = 0; i < R; ++i) {
            const int pos = (warp * R + i) * 32 + lane;
            if (pos < T) {
                const uint64_t k = keys[pos];
                keys[pos] = A.make(L.dom(k), L.gb(k), L.slot(k), L.tok(k));
            }
        }
        L = A;
        __syncthreads();
        radix_sort(keys, hist, T, R, L.slot_at(), L.dom_at() + L.dom_bits, warp_sums);
        int n_dr;
        for_runs(n_dr, n_ur, [&](int i, uint64_t k, bool dh, bool uh, int od, int ou) {
            const int d = L.dom(k);
            p.s.aperm[i] = L.tok(k);
            p.s.sorted_slot[i] = L.slot(k);
            p.s.tok_sc[i] = token_scale(d, L.gb(k));
            if (dh) p.s.d_first[od] = ou;
            if (uh) {
                p.s.a_uptr[ou] = i;
                p.s.a_udom[ou] = d;
                p.s.u_drun[ou] = od + (dh ? 1 : 0) - 1;
            }
        });
        if (tid == 0) p.s.a_uptr[n_ur] = T;
        uptr = p.s.a_uptr;
        udom = p.s.a_udom;
    }
    __syncthreads();  // keys are dead from here; run arrays are visible block-wide

    // 4a. group heads over user runs; a group stays within one domain
    int32_t *grp_first = reinterpret_cast<int32_t *>(keys);  // [n_groups]
    const int Ru = (n_ur + nth - 1) / nth;
    auto group_head = [&](int j) -> bool {
        if (j == 0) return true;
        if (skip0 && j == 1) return true;
        const int dr = p.s.u_drun[j], first = p.s.d_first[dr];  // the domain's first user run
        if (j == first) return true;
        return (j - first - ((skip0 && dr == 0) ? 1 : 0)) % p.umax == 0;
    };
    int ng = 0;
    uint32_t heads = 0;  // this lane's heads, round by round
    for (int i = 0; i < Ru; ++i) {
        const int j = (warp * Ru + i) * 32 + lane;
        const bool h = j < n_ur && group_head(j);
        heads |= (uint32_t)h << i;
        ng += __popc(__ballot_sync(0xffffffffu, h));
    }
    int n_groups;
    int og = block_exclusive_scan(lane == 0 ? ng : 0, &n_groups, warp_sums);
    og = __shfl_sync(0xffffffffu, og, 0);
    for (int i = 0; i < Ru; ++i) {
        const bool h = (heads >> i) & 1u;
        const unsigned m = __ballot_sync(0xffffffffu, h);
        if (h) grp_first[og + __popc(m & ((1u << lane) - 1u))] = (warp * Ru + i) * 32 + lane;
        og += __popc(m);
    }
    __syncthreads();

    // 4b. blocks per group
    const int Eg = (n_groups + nth - 1) / nth;
    const int glo = min(n_groups, tid * Eg), ghi = min(n_groups, glo + Eg);
    auto group_range = [&](int g, int *start, int *len) {
        int a = uptr[grp_first[g]];
        int b = g + 1 < n_groups ? uptr[grp_first[g + 1]] : T;
        *start = a;
        *len = (g == 0 && skip0) ? 0 : b - a;
    };
    int nb = 0;
    for (int g = glo; g < ghi; ++g) {
        int a, len;
        group_range(g, &a, &len);
        nb += (len + TM - 1) / TM;
    }
    int n_blk;
    int ob = block_exclusive_scan(nb, &n_blk, warp_sums);
    for (int g = glo; g < ghi; ++g) {
        int a, len;
        group_range(g, &a, &len);
        int q = (len + TM - 1) / TM;
        int d = udom[grp_first[g]];
        const float sc = d >= 0 ? p.dom_sc[d] : 0.f;
        for (int b = 0; b < q; ++b) {
            int s0 = a + (int)(((int64_t)b * len) / q);
            int s1 = a + (int)(((int64_t)(b + 1) * len) / q);
            int32_t *rec = p.s.blk + (int64_t)BLK_INTS * ob;
            rec[BLK_START] = s0;
            rec[BLK_LEN] = s1 - s0;
            rec[BLK_DOM] = d;
            rec[BLK_RC] = d >= 0 ? p.dom_rc[d] : 0;
            rec[BLK_SC] = __float_as_int(sc);
            ++ob;
        }
    }
    if (tid == 0) {
        p.s.counts[0] = T;
        p.s.counts[1] = n_dseg;
        p.s.counts[2] = n_useg;
        p.s.counts[3] = n_blk;
        max_stack = 0;
    }
    __syncthreads();

    // 5. per-block factor stacks: the residual rows of block b are the rows
    //    of its user runs in order (res_code(slot, rank, k)); each token
    //    records where its own user's rows start.  One warp per block, its
    //    tokens' slots and then their headers loaded together.
    for (int b = warp; b < n_blk; b += SEG_WARPS) {
        const int s0 = p.s.blk[BLK_INTS * b + BLK_START], M = p.s.blk[BLK_INTS * b + BLK_LEN];
        constexpr int NB = TM / 32;
        int slot[NB], rank[NB];
        float su[NB];
#pragma unroll
        for (int i = 0; i < NB; ++i) slot[i] = i * 32 + lane < M ? p.s.sorted_slot[s0 + i * 32 + lane] : -1;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            rank[i] = 0;
            su[i] = 0.f;
            if (slot[i] >= 0) {
                const salt_blob_header *h =
                    reinterpret_cast<const salt_blob_header *>(p.pool + (int64_t)slot[i] * p.slot_stride);
                rank[i] = h->rank;
                su[i] = h->s_u;
            }
        }
        int carry = 0, last_slot = -1;
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const int t = i * 32 + lane;
            int before = __shfl_up_sync(0xffffffffu, slot[i], 1);
            if (lane == 0) before = last_slot;
            last_slot = __shfl_sync(0xffffffffu, slot[i], 31);
            const bool head = t == 0 || slot[i] != before;
            const int contrib = head && slot[i] >= 0 ? rank[i] : 0;
            int incl = contrib;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            if (t < M) {
                const int off = carry + incl - rank[i];
                p.s.tok_uoff[s0 + t] = slot[i] >= 0 ? off : -1;
                p.s.tok_urank[s0 + t] = rank[i];
                p.s.tok_su[s0 + t] = su[i];
                if (contrib > 0)
                    for (int k = 0; k < rank[i]; ++k)
                        if (off + k < S_MAX)
                            p.s.blk_res[(int64_t)b * S_MAX + off + k] = res_code(slot[i], rank[i], k);
            }
            carry += total;
        }
        if (lane == 0) {
            p.s.blk[BLK_INTS * b + BLK_NRES] = carry;
            atomicMax(&max_stack, p.s.blk[BLK_INTS * b + BLK_RC] + carry);
        }
    }
    __syncthreads();
    if (tid == 0) p.s.counts[4] = max_stack;

    // 6. running sum of the expand cost weights over blocks
    const int Eb = (n_blk + nth - 1) / nth;
    const int blo = min(n_blk, tid * Eb), bhi = min(n_blk, blo + Eb);
    auto weight = [&](int b) {
        const int32_t *rec = p.s.blk + (int64_t)BLK_INTS * b;
        return blk_weight(rec[BLK_LEN], rec[BLK_RC] + rec[BLK_NRES]);
    };
    int wsum = 0;
    for (int b = blo; b < bhi; ++b) wsum += weight(b);
    int w_total;
    int wo = block_exclusive_scan(wsum, &w_total, warp_sums);
    for (int b = blo; b < bhi; ++b) {
        wo += weight(b);
        p.s.blk[(int64_t)BLK_INTS * b + BLK_WEND] = wo;
    }
}

}  // namespace

cudaError_t launch_segments(const SegParams &p, cudaStream_t stream)
{
    constexpr size_t hist = (size_t)SEG_WARPS * (1 << RADIX_BITS) * sizeof(uint32_t);
    const size_t smem = (size_t)p.T * sizeof(uint64_t) + hist;
    // the attribute is per device; set it once for each device used
    static unsigned long long configured = 0;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(configured & bit)) {
        e = cudaFuncSetAttribute(seg_build_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(SALT_MAX_TOKENS * sizeof(uint64_t) + hist));
        if (e != cudaSuccess) return e;
        configured |= bit;
    }
    seg_build_kernel<<<1, SEG_THREADS, smem, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace salt
