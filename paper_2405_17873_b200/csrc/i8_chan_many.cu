// Channel-major W4A8 GEMM for layers of several waves: CTA pairs (cta_group::2) walk tiles of 256 channels x up to 256 tokens.
//
// Why.  The two-CTA kernel with the tokens on the rows (i8_pair.cu) is bound by shared memory on int4 weights: 708 cycles per
// k-block of a 256 x 256 tile, of which the tensor pipe needs 512.  With the weights on the M side, expanded straight into
// tensor memory (see i8_chan.cu), a CTA moves per k-block 8 KB of packed rows and 16 KB of token rows in and out of shared
// memory, 384 cycles of the 512.  int8 weights would take the same traffic on either side and stay on i8_pair.cu.
//
// Tensor memory holds the accumulators and the expanded weights.  Tiles of up to 192 tokens have two accumulators, so that a
// tile's epilogue runs beside the next one's main loop, which short reductions need; a tile of 224 or 256 tokens has one and
// waits for its epilogue (some 3000 cycles), which long reductions hide and which buys them the wider tile.
//
// Measured on B200, GEMM alone, before (i8_pair.cu) and now: 1024 x 10240 x 1280 17.9 -> 14.5 us, 4096 x 5120 x 640 23.8 ->
// 18.6, 8192 x 1280 x 1280 18.0 -> 14.3, 3x3 convolutions 4 x 32 x 32 x 1280 -> 1280 54.4 -> 38.2, 4 x 64 x 64 x 640 -> 640
// 46.8 -> 45.0.  A k-block of 192 tokens takes 420 cycles, 384 of them MMA; long layers run at the rate of their tiles' MMAs
// and lose what the last round leaves idle and, at 640 channels, half of the third channel tile.  Short reductions are bound
// by the epilogue, 20 cycles a token (sixteen tokens a turn instead of eight: 14.9 -> 14.3 and 20.2 -> 18.5 us above).
#include <algorithm>

#include "i8_chan.cuh"

namespace mixdq {
namespace i8 {

namespace {

constexpr int GROUPS = 2;                  // of four expansion warps
constexpr int EPI_WARPS = 8;
constexpr int EXP0 = 4, EPI0 = EXP0 + 4 * GROUPS, HELP0 = EPI0 + EPI_WARPS;
// Warps: 0 and 3 MMA issuers (leader), 1 and HELP0 weight producers, 2 and HELP0 + 1 activation producers, expansion, epilogue.
constexpr int THREADS = (HELP0 + 2) * 32;
constexpr int SMEM_MAX = 232448;
// Pairs of k-blocks are numbered through all tiles of a CTA pair; even ones belong to the first warp of each role.
constexpr int NE = 6;                      // pairs whose barriers exist at a time: at least the deepest ring
constexpr int PS = 4;                      // packed slots, a pair each
constexpr int P_BYTES = CH * BK;
constexpr int READY = 0;                   // leader: token rows and expanded weights of both CTAs are in place
constexpr int EMPTY = READY + NE;          // the pair's MMAs have finished
constexpr int FULL_P = EMPTY + NE;
constexpr int EMPTY_P = FULL_P + PS;
constexpr int ACC_FULL = EMPTY_P + PS;     // [2]
constexpr int ACC_EMPTY = ACC_FULL + 2;    // [2], leader
constexpr int GO = ACC_EMPTY + 2;          // leader: the MMA that overwrites the tile's accumulator is issued
constexpr int NUM_BARS = GO + 1;
constexpr int OFF_MISC = NUM_BARS * 8;
constexpr int OFF_P = 1024;                // packed slots, then token rows
constexpr int OFF_X = OFF_P + PS * P_BYTES;
static_assert(OFF_MISC + 16 <= OFF_P && NE % 2 == 0 && PS % 2 == 0, "layout; a waiter must meet every phase of the barriers it waits on");

struct ManyArgs {
    int nt;        // tokens of a tile (multiple of 32)
    int c_tiles;   // tiles along the channels
    int tiles;     // in all
    int bufs;      // accumulators
    int x_pairs, w_pairs;  // ring depths: token rows, expanded weights
    int a_col;     // first tensor-memory column of the expanded weights
    int wide;      // a pair's packed rows are contiguous in memory
};

__global__ void __launch_bounds__(THREADS, 1)
chan_many_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x, const TmaParams p,
                 const ManyArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_MISC + 4);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = cluster_ctarank();
    const bool leader = rank == 0;
    const int pair0 = static_cast<int>(blockIdx.x) >> 1, npairs = static_cast<int>(gridDim.x) >> 1;
    const int my_tiles = (g.tiles - pair0 + npairs - 1) / npairs;
    const int nkb = p.k_blocks, pairs = (nkb + 1) >> 1, rows = g.nt >> 1;
    const uint32_t x_bytes = static_cast<uint32_t>(rows) * BK;
    const uint32_t bar0 = smem_u32(smem), p0 = bar0 + OFF_P, x0 = bar0 + OFF_X;
    const uint32_t lead_bar0 = map_to_cta(bar0, 0);

    pdl_launch_dependents();
    if (warp == 3 && lane == 0) {
        for (int s = 0; s < NE; ++s) {
            mbar_init(bar0 + 8 * (READY + s), 1 + 2 * 4);  // activation bytes; a group's four warps of both CTAs
            mbar_init(bar0 + 8 * (EMPTY + s), 1);
        }
        for (int s = 0; s < PS; ++s) {
            mbar_init(bar0 + 8 * (FULL_P + s), 1);
            mbar_init(bar0 + 8 * (EMPTY_P + s), 4);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar0 + 8 * (ACC_FULL + b), 2);  // one commit of each issuer
            mbar_init(bar0 + 8 * (ACC_EMPTY + b), 2 * EPI_WARPS);
        }
        mbar_init(bar0 + 8 * GO, 1);
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;
        fence_barrier_init();
    } else if (warp == 0) {
        tmem_alloc_pair(smem_u32(s_tmem), 512);
        tmem_relinquish_pair();
    } else if (warp == 1 && lane == 0) {
        tma_prefetch_desc(&tmap_w);
    } else if (warp == 2 && lane == 0) {
        tma_prefetch_desc(&tmap_x);
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync();  // no CTA signals a barrier of its peer before that barrier exists
    tc_fence_after_sync();
    constexpr uint32_t tmem_base = 0;  // all 512 columns are this CTA's
    if (*s_tmem != tmem_base) *abort_flag = 1;
    // the weights are constants of the layer: their producers and the warps that expand them run ahead of earlier kernels
    const bool expander = warp >= EXP0 && warp < EPI0;
    if (warp != 1 && warp != HELP0 && !expander) pdl_wait();

    if (warp == 0 || warp == 3) {
        // ------------------------------------------------------------ MMA issuers (two warps of the leader)
        // They take alternate pairs into one accumulator, after the MMA that overwrites it (see i8_chan.cu).
        if (leader) {
            const uint32_t idesc = make_idesc(2, 1, 2 * CH, static_cast<uint32_t>(g.nt));
            const uint64_t x_desc0 = smem_desc_sw128(x0);
            const int which = warp == 0 ? 0 : 1;
            int sx = which % g.x_pairs, sw = which % g.w_pairs, sb = which;
            uint32_t par = 0;
            bool ok = true;
            for (int t = 0; t < my_tiles; ++t) {
                const int buf = g.bufs == 2 ? t & 1 : 0, use = g.bufs == 2 ? t >> 1 : t;
                const uint32_t acc = tmem_base + buf * g.nt;
                const int first = (which + t * pairs) & 1;  // of this warp's pairs in the tile
                if (first == 0)
                    ok = ok && mbar_wait(bar0 + 8 * (ACC_EMPTY + buf), (use & 1) ^ 1, abort_flag);
                else if (first < pairs)
                    ok = ok && mbar_wait(bar0 + 8 * GO, t & 1, abort_flag);
                for (int j = first; j < pairs; j += 2) {
                    ok = ok && mbar_wait(bar0 + 8 * (READY + sb), par, abort_flag);
                    if (!__all_sync(0xffffffffu, ok)) break;
                    tc_fence_after_sync();
                    const uint64_t x_desc = x_desc0 + static_cast<uint32_t>(2 * sx) * (x_bytes >> 4);
                    const uint32_t a = tmem_base + g.a_col + sw * 64;
                    const bool both = 2 * j + 1 < nkb;
                    if (elect_one()) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            if (h == 1 && !both) break;
                            const uint64_t xd = x_desc + h * (x_bytes >> 4);
#pragma unroll
                            for (int k = 0; k < BK / 32; ++k)
                                mma_i8_ts<2>(acc, a + 32 * h + 8 * k, xd + 2 * k, idesc, (j != 0 || h != 0 || k != 0) ? 1u : 0u);
                        }
                        if (j == 0) {
                            tc_fence_before_sync();
                            mbar_arrive(bar0 + 8 * GO);
                        }
                        tc_commit_pair(bar0 + 8 * (EMPTY + sb), 3);
                    }
                    __syncwarp();
                    sx += 2;
                    while (sx >= g.x_pairs) sx -= g.x_pairs;
                    sw += 2;
                    while (sw >= g.w_pairs) sw -= g.w_pairs;
                    sb += 2;
                    if (sb >= NE) {
                        sb -= NE;
                        par ^= 1;
                    }
                }
                if (!__all_sync(0xffffffffu, ok)) break;
                if (elect_one()) tc_commit_pair(bar0 + 8 * (ACC_FULL + buf), 3);  // (none in this tile: nothing to wait for)
                __syncwarp();
            }
        }
    } else if (warp == 1 || warp == HELP0) {
        // ------------------------------------------------------------ packed weight rows of this CTA's channels
        const int which = warp == 1 ? 0 : 1;
        int s = which;
        uint32_t par = 1;  // slots start out free
        bool ok = true;
        for (int t = 0; t < my_tiles && ok; ++t) {
            const int tile = pair0 + t * npairs;
            const int n0 = (tile % g.c_tiles) * (2 * CH) + static_cast<int>(rank) * CH;
            const int first = (which + t * pairs) & 1;
            const int end = p.test_drop_b_kblock && t == my_tiles - 1 ? (p.test_drop_b_kblock - 1) >> 1 : pairs;
            KPos at(2 * first, p.cblocks);
            for (int j = first; j < end; j += 2) {
                ok = mbar_wait(bar0 + 8 * (EMPTY_P + s), par, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const bool both = 2 * j + 1 < nkb;
                    const uint32_t full = bar0 + 8 * (FULL_P + s), dst = p0 + s * P_BYTES;
                    mbar_arrive_expect_tx(full, (g.wide || both) ? P_BYTES : P_BYTES / 2);
                    tma_load_2d(dst, &tmap_w, (at.tap * p.Cin + at.c * BK) >> 1, n0, full);
                    if (!g.wide && both) {
                        KPos next = at;
                        next.advance(1, p.cblocks);
                        tma_load_2d(dst + P_BYTES / 2, &tmap_w, (next.tap * p.Cin + next.c * BK) >> 1, n0, full);
                    }
                }
                __syncwarp();
                at.advance(4, p.cblocks);
                s += 2;
                if (s >= PS) {
                    s -= PS;
                    par ^= 1;
                }
            }
        }
    } else if (warp == 2 || warp == HELP0 + 1) {
        // ------------------------------------------------------------ int8 token rows (this CTA's half of the tile's)
        const int which = warp == 2 ? 0 : 1;
        int s = which % g.x_pairs, sb = which;  // slot and barrier of the pair
        int qb = which - g.x_pairs;             // barrier of the pair whose MMAs free the slot (negative: the first lap)
        uint32_t qpar = 0;
        bool ok = true;
        for (int t = 0; t < my_tiles && ok; ++t) {
            const int tile = pair0 + t * npairs;
            const int m0 = (tile / g.c_tiles) * g.nt + static_cast<int>(rank) * rows;
            int img = 0, wi = 0, hi = 0;
            if (p.conv) {
                const int mc = m0 < p.M ? m0 : 0;  // no output rows: any pixels will do
                img = mc / p.HoWo;
                const int rem = mc - img * p.HoWo;
                const int ho = rem / p.Wo;
                hi = p.stride * ho - 1 + p.pad;
                wi = p.stride * (rem - ho * p.Wo) - 1 + p.pad;
            }
            const int first = (which + t * pairs) & 1;
            KPos at(2 * first, p.cblocks);
            for (int j = first; j < pairs; j += 2) {
                if (qb >= 0) ok = mbar_wait(bar0 + 8 * (EMPTY + qb), qpar, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                if (elect_one()) {
                    const int n = 2 * j + 1 < nkb ? 2 : 1;
                    if (leader) mbar_arrive_expect_tx(bar0 + 8 * (READY + sb), n * 2 * x_bytes);
                    const uint32_t full = lead_bar0 + 8 * (READY + sb);
                    KPos pos = at;
                    for (int h = 0; h < n; ++h) {
                        const uint32_t dst = x0 + (2 * s + h) * x_bytes;
                        if (p.conv) {
                            const int kh = pos.tap / 3, kw = pos.tap - 3 * kh;
                            tma_load_im2col_pair(dst, &tmap_x, pos.c * BK, wi, hi, img, kw, kh, full);
                        } else {
                            tma_load_2d_pair(dst, &tmap_x, pos.c * BK, m0, full);
                        }
                        pos.advance(1, p.cblocks);
                    }
                }
                __syncwarp();
                at.advance(4, p.cblocks);
                s += 2;
                while (s >= g.x_pairs) s -= g.x_pairs;
                sb += 2;
                if (sb >= NE) sb -= NE;
                qb += 2;
                if (qb >= NE) {
                    qb -= NE;
                    qpar ^= 1;
                }
            }
        }
    } else if (expander) {
        // ------------------------------------------------------------ packed int4 -> int8 (x16) in tensor memory
        const int group = (warp - EXP0) >> 2;
        const uint32_t a_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + g.a_col;
        const PackedRows rows_of((warp & 3) * 32 + lane, g.wide);
        const int total = my_tiles * pairs;
        uint4 w[8];
        int sw = group % g.w_pairs, sb = group;
        int sp = group;                   // packed slot of the next fetch and its phase
        uint32_t ppar = 0;
        int qb = group - g.w_pairs;       // barrier of the pair whose MMAs free the slot (negative: the first lap), its phase
        uint32_t qpar = 0;
        auto fetch = [&]() {
            const bool ok = mbar_wait(bar0 + 8 * (FULL_P + sp), ppar, abort_flag);
            rows_of.load(smem + OFF_P + sp * P_BYTES, w);
            return ok;
        };
        int j = group % pairs;
        bool ok = group < total ? fetch() : true;
        for (int q = group; q < total; q += GROUPS) {
            if (ok && qb >= 0) ok = mbar_wait(bar0 + 8 * (EMPTY + qb), qpar, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) break;  // the warp leaves together
            tc_fence_after_sync();
            expand_row(w, a_lane + sw * 64);
            if (2 * j + 1 < nkb) expand_row(w + 4, a_lane + sw * 64 + 32);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar0 + 8 * (EMPTY_P + sp));
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(lead_bar0 + 8 * (READY + sb));
            sp += GROUPS;
            if (sp >= PS) {
                sp -= PS;
                ppar ^= 1;
            }
            if (q + GROUPS < total) ok = fetch();
            sw += GROUPS;
            while (sw >= g.w_pairs) sw -= g.w_pairs;
            sb += GROUPS;
            if (sb >= NE) sb -= NE;
            qb += GROUPS;
            if (qb >= NE) {
                qb -= NE;
                qpar ^= 1;
            }
            j += GROUPS;
            while (j >= pairs) j -= pairs;
        }
        pdl_wait();
    } else {
        // ------------------------------------------------------------ epilogue: eight warps
        const int ew = warp - EPI0;
        const bool pairs_ok = ((p.N | static_cast<int>(p.ldy)) & 1) == 0 && (reinterpret_cast<uintptr_t>(p.Y) & 3) == 0;
        const float sx = p.act_scale ? ld_pinned(p.act_scale) : 0.f;
        const int zshift = p.act_zero ? 128 - __ldg(p.act_zero) : 0;
        for (int t = 0; t < my_tiles; ++t) {
            const int tile = pair0 + t * npairs;
            const int tok0 = (tile / g.c_tiles) * g.nt;
            const int n = (tile % g.c_tiles) * (2 * CH) + static_cast<int>(rank) * CH + (warp & 3) * 32 + lane;  // this lane's channel
            const int buf = g.bufs == 2 ? t & 1 : 0, use = g.bufs == 2 ? t >> 1 : t;
            float comb = 0.f, bias = 0.f;
            int zterm = 0;  // (128 - zero) * sum of the channel's weight codes
            if (n < p.N) {
                if (p.act_zero) zterm = zshift * __ldg(p.w_code_sums + n);
                if (p.w_scale) {
                    comb = sx * ld_pinned(p.w_scale + n);
                    if (p.bias) bias = __half2float(p.bias[n]);
                    if (p.act_zero) bias = fmaf(static_cast<float>(zterm), comb, bias);
                }
            }
            comb *= 0.0625f;  // the sums carry the factor 16 of the nibble placement: an exact power of two
            // one warp polls, the others sleep in a named barrier (polling loads the producers' path)
            // and the same barrier carries its verdict, so that all eight warps take the same path
            const bool ok = ew != 0 || mbar_wait(bar0 + 8 * (ACC_FULL + buf), use & 1, abort_flag);
            __syncwarp();
            uint32_t go;
            asm volatile(
                "{\n\t"
                ".reg .pred p, q;\n\t"
                "setp.ne.u32 q, %1, 0;\n\t"
                "barrier.cta.red.and.pred p, 1, %2, q;\n\t"
                "selp.u32 %0, 1, 0, p;\n\t"
                "}\n"
                : "=r"(go)
                : "r"(ok ? 1u : 0u), "n"(32 * EPI_WARPS)
                : "memory");
            if (!go) break;
            tc_fence_after_sync();
            const uint32_t acc = tmem_base + buf * g.nt + (static_cast<uint32_t>((warp & 3) * 32) << 16);
            const int cols = min(g.nt, p.M - tok0);
            if (p.Y && pairs_ok && !p.acc_out) {
                store_tokens<ACC_INT, 16>(acc, 0, (ew >> 2) * 16, 32, cols, comb, 0.f, bias, p.Y + (n & ~1), p.ldy, tok0, p.M, n < p.N, false,
                                    lane);
            } else {
                // odd widths, and the raw sums of the parity hook
                for (int c0 = (ew >> 2) * 8; c0 < cols; c0 += 16) {
                    uint32_t r[8];
                    tmem_ld_32x8(acc + c0, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int m = tok0 + c0 + i;
                        if (m >= p.M || n >= p.N) continue;
                        const int32_t a = static_cast<int32_t>(r[i]);
                        if (p.acc_out) p.acc_out[static_cast<long long>(m) * p.N + n] = (a >> 4) + zterm;
                        if (p.Y) p.Y[m * p.ldy + n] = __float2half_rn(fmaf(__int2float_rn(a), comb, bias));
                    }
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(lead_bar0 + 8 * (ACC_EMPTY + buf));
        }
    }

    report_abandoned_wait(abort_flag, p.status);
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync();  // neither CTA leaves while its peer may still signal its barriers or use its memory
    if (warp == 0) tmem_dealloc_pair(tmem_base, 512);
}

}  // namespace

// (Two pairs of k-blocks at least: with one, an MMA issuer could run a tile ahead of the other.)
bool chan_many_tile_ok(int tokens, int k_blocks) { return tokens >= 32 && tokens % 32 == 0 && tokens <= 256 && k_blocks >= 3; }

// codes: as for run_chan; W4 only, any linear layer or 3x3 convolution.
int run_chan_many(const Params& p, int amode, const void* packed, const int8_t* codes, int tokens, int num_sms, cudaStream_t stream)
{
    const bool conv = amode == A_CONV3;
    const int pad = (conv && p.act_zero) ? 1 : 0;
    const int cin = conv ? p.Cin : p.K, rows = tokens / 2;
    TmaParams tp{};
    tp.M = p.M;
    tp.N = p.N;
    tp.act_scale = p.act_scale;
    tp.act_zero = p.act_zero;
    tp.w_code_sums = p.w_code_sums;
    tp.w_scale = p.w_scale;
    tp.bias = p.bias;
    tp.Y = p.Y;
    tp.ldy = p.ldy;
    tp.acc_out = p.acc_out;
    tp.status = p.status;
    tp.test_drop_b_kblock = p.test_drop_b_kblock;
    tp.cblocks = static_cast<int>(ceil_div(cin, BK));
    tp.k_blocks = (conv ? 9 : 1) * tp.cblocks;
    if (!chan_many_tile_ok(tokens, tp.k_blocks) || amode == A_BOS || p.addend) return MIXDQ_ERR_INVALID_ARG;
    if (conv) {
        tp.conv = 1;
        tp.pad = pad;
        tp.stride = p.stride;
        tp.Cin = p.Cin;
        tp.HoWo = p.Ho * p.Wo;
        tp.Wo = p.Wo;
    }
    ManyArgs g{};
    g.nt = tokens;
    g.c_tiles = static_cast<int>(ceil_div(p.N, 2 * CH));
    g.tiles = g.c_tiles * static_cast<int>(ceil_div(p.M, tokens));
    g.bufs = tokens <= 192 ? 2 : 1;
    g.a_col = g.bufs == 2 ? 2 * tokens : 256;
    g.w_pairs = std::min(4, (512 - g.a_col) / 64);
    const int x_bytes = rows * BK;
    g.x_pairs = std::min(NE, (SMEM_MAX - OFF_X) / (2 * x_bytes)) & ~1;  // (even: see launch_t of i8_chan.cu)
    g.wide = !conv || cin % BK == 0;
    CUtensorMap tw, tx;
    const int rc = encode_chan_branch(&tw, &tx, p, conv, pad, cin, packed, true, g.wide, codes, rows);
    if (rc != MIXDQ_OK) return rc;
    if (ensure_dynamic_smem(reinterpret_cast<const void*>(chan_many_kernel), SMEM_MAX) != MIXDQ_OK) return MIXDQ_ERR_CUDA;
    const int npairs = std::min(num_sms / 2, g.tiles);
    return launch_pdl_cluster(chan_many_kernel, dim3(static_cast<unsigned>(2 * npairs)), dim3(THREADS),
                              static_cast<size_t>(OFF_X + g.x_pairs * 2 * x_bytes), stream, 2u, 1u, tw, tx, tp, g);
}

}  // namespace i8
}  // namespace mixdq
