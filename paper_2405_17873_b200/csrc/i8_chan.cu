// Channel-major W8A8 / W4A8 GEMM: the WEIGHTS are the 128-row operand of the tensor-core instruction (one output channel
// per lane of tensor memory) and the tokens its N side.
//
// Why.  The kernels with tokens on the rows (i8_tma.cu, i8_pair.cu) are bound by shared-memory bandwidth, 128 bytes per
// cycle and SM: per k-block of 128 an activation tile of 128 rows is written and read (32 KB = 256 cycles), and an int4
// weight row of 64 bytes is written, read, written again as 128 bytes of int8 and read by the MMA (384 bytes = 3 cycles
// per row) -- the per-k-block costs measured for the two-CTA kernel, 350 + 1.4 bn cycles with int4 and 250 + 1.2 bn
// with int8 weights, are these sums.  And a layer of few tokens has few 128-row tiles.  With the weights on the M side
//   * int4 weights are expanded to int8 straight into TENSOR MEMORY, which the MMA reads as its A operand: a packed row
//     costs shared memory one write and one read of 64 bytes, so a 128-channel k-block costs 128 cycles instead of 384;
//   * the token count of a tile is free in steps of 16, so a layer of few tokens still covers the SMs;
//   * two CTAs (CG = 2) share a tile of 256 channels: each holds its own channels' weights and HALF of the tokens.
//
// One tile per CTA (pair).  What bounds the layers this form is for (one wave of tiles, ten to forty k-blocks) is the chain
// grid completion -> first loads -> main loop -> epilogue, and in it the LATENCY of a ring slot (TMA request to the slot's
// return: some 1900 cycles), so the rings are as deep as the SM allows: the weights are constants of the layer, and up to
// twelve k-blocks of them are loaded and expanded (384 columns of tensor memory) while the quantization pass still runs;
// when that has finished, up to twelve activation tiles are requested at once and the MMAs follow their arrival.
//
// The int8 codes arrive by TMA: linear rows, or an im2col map of the image (any number of consecutive output pixels at one
// filter tap).
//
// Measured on B200, GEMM alone in a chain of launches, against the forms with tokens on the rows: W4 1024 x 1280 x 1280 5.0
// us (6.5), 1024 x 1280 x 5120 9.5 (14.7), 256 x 1280 x 1280 3.5 (7.0), 616 x 1280 x 2048 5.1 (8.8), 4096 x 640 x 640 6.3
// (7.9), 3x3 convolution 48 x 48 x 640 -> 640 10.6 (16.7), 4 x 16 x 16 x 640 -> 1280 10.3 (16.9); W8 5.2 (5.6), 10.0 (11.9),
// 3.9 (6.7), 5.5 (8.3), 6.3 (6.5), 11.4 (15.3), 10.8 (15.4).  A long reduction takes 270 cycles per k-block of 128 channels x
// 80 tokens, of which the tensor pipe is busy 160: two issuers, each some 1000 cycles per pair (wait 150, eight MMAs and a
// commit 450, the loop), and two activation producers of about the same are the next limits; four of either gained nothing.
//
// Epilogue: a thread owns a channel, so scale and bias live in two registers; neighbouring lanes swap halves of a packed
// token pair and store channel pairs, 64 contiguous bytes of an output row per warp -- no staging tile.
#include <algorithm>
#include <cmath>

#include "i8_chan.cuh"

namespace mixdq {
namespace i8 {

namespace {

constexpr int TOK_MAX = 256;   // tokens of a tile
constexpr int ROWS_MAX = 128;  // token rows of one CTA
constexpr int EXP_GROUPS = 3;  // of four warps: expansion (W4), then epilogue
constexpr int WORKERS = 4 * EXP_GROUPS, WORK0 = 4, HELP0 = WORK0 + WORKERS;
constexpr int THREADS = (HELP0 + 2) * 32;
constexpr int SMEM_MAX = 232448;

// Warps: 0 MMA issuer and tensor-memory allocation, 1 and 16 weight producers, 2 and 17 activation producers, 3 barrier
// set-up, then second MMA issuer; 4 .. 15 expansion (W4), three groups of four, then the epilogue.
template <int CG, bool W4>
struct Chan {
    static constexpr int W_BYTES = CH * BK;        // int8 weight rows of a k-block (W8)
    static constexpr int P_BYTES = CH * BK;        // packed int4 weight rows of two k-blocks
    static constexpr int ISSUERS = 2;
    // k-blocks go through in pairs: one barrier says that a pair's tiles are in place, one commit that its MMAs have
    // finished, which frees the pair's slots of all rings.  Ring depths in k-blocks; run-time ones: activation slots, and
    // W4's slots in tensor memory, 12 beside an accumulator of up to 128 tokens, 8 beside a wider one.
    static constexpr int NE = 6;                   // pairs whose barriers exist at a time: at least the deepest ring
    static constexpr int XS_MAX = 2 * NE;
    static constexpr int WS_MAX = W4 ? 12 : 8;
    static constexpr int PS = W4 ? 6 : 0;          // packed rows: slots of a pair each
    // (a waiter must meet every phase of the barriers it waits on: expansion groups those of every third pair)
    static_assert(NE % EXP_GROUPS == 0 && PS % EXP_GROUPS == 0 && PS <= NE, "barriers and groups");
    static constexpr int OFF_W = 0;
    static constexpr int RING_W = W4 ? PS * P_BYTES : WS_MAX * W_BYTES;
    static constexpr int READY = 0;                   // leader: the pair's token rows and weights of both CTAs are in place
    static constexpr int EMPTY = READY + NE;          // the MMAs of the pair have finished
    static constexpr int FULL_P = EMPTY + NE;         // W4: packed rows landed
    static constexpr int EMPTY_P = FULL_P + PS;       // W4: packed rows read
    static constexpr int ACC_FULL = EMPTY_P + PS;
    static constexpr int GO = ACC_FULL + 1;           // leader: the MMA that overwrites the accumulator is issued
    static constexpr int GO2 = GO + 1;                // the same for the second branch's
    static constexpr int NUM_BARS = GO2 + 1;
    static constexpr int OFF_BARS = RING_W;
    static constexpr int OFF_MISC = OFF_BARS + NUM_BARS * 8;
    static constexpr int OFF_X = (OFF_MISC + 16 + 1023) & ~1023;
};

struct ChanArgs {
    int nt;        // tokens of a tile (multiple of 16 CG)
    int c_tiles;   // channel tiles (128 CG channels each)
    int x_slots, w_slots;
    int a_col;     // W4: first tensor-memory column of the expanded weights
    int wide;      // W4: a pair's packed rows are contiguous in memory and arrive as 128-byte rows
    // two branches (shortcut-splitting, Sec. 4.1): the k-blocks from kb_lo on are the second branch's, with maps, geometry,
    // scale and accumulator (column acc2) of its own; acc_out2: its sums (parity hook)
    int kb_lo, cblocks2, Cin2, acc2;
    const float* act_scale2;
    int32_t* acc_out2;
};

// Waits until the MMAs of the pair of k-block `was` have finished.
template <class L>
__device__ __forceinline__ bool wait_mmas(uint32_t bar0, int was, volatile int* abort_flag)
{
    const uint32_t q = static_cast<uint32_t>(was) >> 1;
    return mbar_wait(bar0 + 8 * (L::EMPTY + q % L::NE), (q / L::NE) & 1, abort_flag);
}

// Grid: CG CTAs (a cluster) per tile of 128 CG channels x nt tokens, channel tiles fastest.
template <int CG, bool W4, bool TWO>
__global__ void __launch_bounds__(THREADS, 1)
chan_gemm_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x,
                 const __grid_constant__ CUtensorMap tmap_w2, const __grid_constant__ CUtensorMap tmap_x2, const TmaParams p,
                 const ChanArgs g)
{
    using L = Chan<CG, W4>;
    extern __shared__ __align__(1024) uint8_t smem[];
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::OFF_MISC + 4);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
    const bool leader = rank == 0;
    const int tile = static_cast<int>(blockIdx.x) / CG;
    const Pairs<TWO> pr(p.k_blocks, g.kb_lo);
    const int pairs = pr.n, rows = g.nt / CG;  // token rows this CTA holds
    const int tok0 = (tile / g.c_tiles) * g.nt;
    const int n0 = (tile % g.c_tiles) * (CG * CH) + static_cast<int>(rank) * CH;
    const uint32_t x_bytes = static_cast<uint32_t>(rows) * BK;

    const uint32_t bar0 = smem_u32(smem + L::OFF_BARS);
    const uint32_t x0 = smem_u32(smem + L::OFF_X), w0 = smem_u32(smem + L::OFF_W);
    const uint32_t lead_bar0 = CG == 2 ? map_to_cta(bar0, 0) : bar0;

    pdl_launch_dependents();
    if (warp == 3 && lane == 0) {
        for (int s = 0; s < L::NE; ++s) {
            mbar_init(bar0 + 8 * (L::READY + s), 1 + (W4 ? CG * 4 : 1));  // activation bytes; weight bytes or expansion warps
            mbar_init(bar0 + 8 * (L::EMPTY + s), 1);
        }
        for (int s = 0; s < L::PS; ++s) {
            mbar_init(bar0 + 8 * (L::FULL_P + s), 1);
            mbar_init(bar0 + 8 * (L::EMPTY_P + s), 4);
        }
        mbar_init(bar0 + 8 * L::ACC_FULL, L::ISSUERS);
        mbar_init(bar0 + 8 * L::GO, 1);
        mbar_init(bar0 + 8 * L::GO2, 1);
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;  // the swizzled tiles need the alignment the array is declared with
        fence_barrier_init();
    } else if (warp == 0) {
        if (CG == 1) {
            tmem_alloc(smem_u32(s_tmem), 512);
            tmem_relinquish();
        } else {
            tmem_alloc_pair(smem_u32(s_tmem), 512);
            tmem_relinquish_pair();
        }
    } else if (warp == 1 && lane == 0) {
        tma_prefetch_desc(&tmap_w);
    } else if (warp == 2 && lane == 0) {
        tma_prefetch_desc(&tmap_x);
    }
    tc_fence_before_sync();
    __syncthreads();
    if (CG == 2) cluster_sync();  // no CTA signals a barrier of its peer before that barrier exists
    tc_fence_after_sync();
    // all 512 columns are this CTA's, so its tensor memory starts at address 0: a constant, which the MMA issue relies on
    constexpr uint32_t tmem_base = 0;
    if (*s_tmem != tmem_base) *abort_flag = 1;
    // the weights are constants of the layer: their producer and the warps that expand them run ahead of earlier kernels
    const bool expander = W4 && warp >= WORK0 && warp < HELP0;
    if (warp != 1 && warp != HELP0 && !expander) pdl_wait();

    if (warp == 0 || warp == 3) {
        // ------------------------------------------------------------ MMA issuers (two warps of the leader)
        // One k-block at a time cost its issuer some 430 cycles: four MMAs and a commit 160 to 190, the probe of its barrier
        // 100, the rest the loop.  So the k-blocks come in pairs, and two warps take alternate pairs into ONE accumulator
        // (integer sums: the order does not matter), after the MMA that overwrites it.  (Four warps got in each other's way:
        // the instructions enter the tensor pipe no faster than one every 45 cycles.)
        // A whole warp runs the loop and one elected lane issues: descriptors and addresses then stay in uniform registers
        // (a lane that runs alone needs twice the time).
        if (leader) {
            const uint32_t idesc = make_idesc(2, 1, CG * CH, static_cast<uint32_t>(g.nt));
            const uint64_t w_desc0 = smem_desc_sw128(w0), x_desc0 = smem_desc_sw128(x0);
            const int first = warp == 0 ? 0 : 1;
            int sx = 2 * first % g.x_slots, sw = 2 * first, sb = first;
            uint32_t par = 0;
            bool ok = first == 0 || first >= pairs || mbar_wait(bar0 + 8 * L::GO, 0, abort_flag);
            for (int j = first; j < pairs; j += L::ISSUERS) {
                ok = ok && mbar_wait(bar0 + 8 * (L::READY + sb), par, abort_flag);
                if (TWO && j == pr.lo + 1) ok = ok && mbar_wait(bar0 + 8 * L::GO2, 0, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                tc_fence_after_sync();
                const uint64_t x_desc = x_desc0 + static_cast<uint32_t>(sx) * (x_bytes >> 4);
                const uint64_t w_desc = w_desc0 + sw * (L::W_BYTES >> 4);
                const bool both = pr.both(j);
                const bool fresh = j == 0 || (TWO && j == pr.lo);  // overwrites its accumulator
                const uint32_t acc = tmem_base + (pr.second(j) ? g.acc2 : 0);
                if (elect_one()) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && !both) break;
                        const uint64_t xd = x_desc + h * (x_bytes >> 4);
#pragma unroll
                        for (int k = 0; k < BK / 32; ++k) {
                            const uint32_t add = (!fresh || h != 0 || k != 0) ? 1u : 0u;
                            const uint64_t wd = w_desc + h * (L::W_BYTES >> 4) + 2 * k;
                            if (W4)
                                mma_i8_ts<CG>(acc, tmem_base + g.a_col + sw * 32 + 32 * h + 8 * k, xd + 2 * k, idesc, add);
                            else if (CG == 1)
                                mma_i8_ss(acc, wd, xd + 2 * k, idesc, add);
                            else
                                mma_i8_pair(acc, wd, xd + 2 * k, idesc, add);
                        }
                    }
                    if (fresh) {
                        tc_fence_before_sync();
                        mbar_arrive(bar0 + 8 * (j == 0 ? L::GO : L::GO2));
                    }
                    commit_mmas<CG>(bar0 + 8 * (L::EMPTY + sb));
                    if (j + L::ISSUERS >= pairs) commit_mmas<CG>(bar0 + 8 * L::ACC_FULL);
                }
                __syncwarp();
                sx += 2 * L::ISSUERS;
                while (sx >= g.x_slots) sx -= g.x_slots;
                sw += 2 * L::ISSUERS;
                if (sw >= g.w_slots) sw -= g.w_slots;
                sb += L::ISSUERS;
                if (sb >= L::NE) {
                    sb -= L::NE;
                    par ^= 1;
                }
            }
            if (first >= pairs && elect_one()) commit_mmas<CG>(bar0 + 8 * L::ACC_FULL);  // (nothing to wait for)
            __syncwarp();
        }
    } else if (warp == 1 || warp == HELP0) {
        // ------------------------------------------------------------ weight rows of this CTA's channels
        auto request = [&](int s, int sb, int u, KPos at) {  // a pair of k-blocks
            const int n = pr.both(u) ? 2 : 1;
            const bool second = pr.second(u);
            const CUtensorMap* map = second ? &tmap_w2 : &tmap_w;
            const int cblocks = second ? g.cblocks2 : p.cblocks, cin = second ? g.Cin2 : p.Cin;
            auto x_of = [&](const KPos& at) { return at.tap * cin + at.c * BK; };  // first reduction index of a k-block
            if (W4) {  // on a barrier of its own
                const uint32_t full = bar0 + 8 * (L::FULL_P + s), dst = w0 + s * L::P_BYTES;
                mbar_arrive_expect_tx(full, (g.wide || n == 2) ? L::P_BYTES : L::P_BYTES / 2);
                tma_load_2d(dst, map, x_of(at) >> 1, n0, full);
                if (!g.wide && n == 2) {
                    at.advance(1, cblocks);
                    tma_load_2d(dst + L::P_BYTES / 2, map, x_of(at) >> 1, n0, full);
                }
            } else {
                if (leader) mbar_arrive_expect_tx(bar0 + 8 * (L::READY + sb), n * CG * L::W_BYTES);
                for (int h = 0; h < n; ++h) {
                    const uint32_t dst = w0 + (2 * s + h) * L::W_BYTES;
                    if (CG == 1)
                        tma_load_2d(dst, map, x_of(at), n0, bar0 + 8 * (L::READY + sb));
                    else
                        tma_load_2d_pair(dst, map, x_of(at), n0, lead_bar0 + 8 * (L::READY + sb));
                    at.advance(1, cblocks);
                }
            }
        };
        produce<TWO>(warp == 1 ? 0 : 1, lane, W4 ? L::PS : L::WS_MAX / 2, pr, p.cblocks, g.cblocks2,
                     bar0 + 8 * (W4 ? L::EMPTY_P : L::EMPTY), W4 ? L::PS : L::NE, abort_flag, request);
    } else if (warp == 2 || warp == HELP0 + 1) {
        // ------------------------------------------------------------ int8 token rows by TMA
        const int m0 = tok0 + static_cast<int>(rank) * rows;
        int img = 0, wi = 0, hi = 0;
        if (p.conv) {
            const int mc = m0 < p.M ? m0 : 0;  // no output rows: any pixels will do
            img = mc / p.HoWo;
            const int rem = mc - img * p.HoWo;
            const int ho = rem / p.Wo;
            hi = p.stride * ho - 1 + p.pad;
            wi = p.stride * (rem - ho * p.Wo) - 1 + p.pad;
        }
        auto request = [&](int s, int sb, int u, KPos at) {
            const uint32_t full = bar0 + 8 * (L::READY + sb), lead_full = lead_bar0 + 8 * (L::READY + sb);
            const int n = pr.both(u) ? 2 : 1;
            const bool second = pr.second(u);
            const CUtensorMap* map = second ? &tmap_x2 : &tmap_x;
            if (leader) mbar_arrive_expect_tx(full, n * CG * x_bytes);
            for (int h = 0; h < n; ++h) {
                const uint32_t dst = x0 + (2 * s + h) * x_bytes;
                if (p.conv) {
                    const int kh = at.tap / 3, kw = at.tap - 3 * kh;
                    if (CG == 1)
                        tma_load_im2col(dst, map, at.c * BK, wi, hi, img, kw, kh, full);
                    else
                        tma_load_im2col_pair(dst, map, at.c * BK, wi, hi, img, kw, kh, lead_full);
                } else if (CG == 1) {
                    tma_load_2d(dst, map, at.c * BK, m0, full);
                } else {
                    tma_load_2d_pair(dst, map, at.c * BK, m0, lead_full);
                }
                at.advance(1, second ? g.cblocks2 : p.cblocks);
            }
        };
        produce<TWO>(warp == 2 ? 0 : 1, lane, g.x_slots / 2, pr, p.cblocks, g.cblocks2, bar0 + 8 * L::EMPTY, L::NE, abort_flag, request);
    } else if (expander) {
        // ------------------------------------------------------------ packed int4 -> int8 (x16) in tensor memory
        // A thread owns a channel: its 64 packed bytes of a k-block become 32 columns of its lane.  Groups of four warps
        // take alternate pairs and fetch the next packed rows into registers before they wait for its slots.  (One k-block at
        // a time, a turn took its group 1200 cycles, half of them for the waits and arrivals.)  The swizzle of the rows (128
        // bytes, or 64 where a pair is not contiguous) makes the reads conflict-free.
        const int group = (warp - WORK0) >> 2, row = (warp & 3) * 32 + lane;
        constexpr uint32_t PS = L::PS > 0 ? L::PS : 1;
        const uint32_t a_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + g.a_col;
        const PackedRows rows_of(row, g.wide);
        int sw = 2 * group;  // slot of the pair's first k-block
        if (sw >= g.w_slots) sw -= g.w_slots;
        uint4 w[8];
        auto fetch = [&](int j) {
            const uint32_t q = static_cast<uint32_t>(j), sp = q % PS;
            const bool ok = mbar_wait(bar0 + 8 * (L::FULL_P + sp), (q / PS) & 1, abort_flag);
            rows_of.load(smem + L::OFF_W + sp * L::P_BYTES, w);
            return ok;
        };
        bool ok = group < pairs ? fetch(group) : true;
        for (int j = group; j < pairs; j += EXP_GROUPS) {
            if (ok && 2 * j >= g.w_slots) ok = wait_mmas<L>(bar0, 2 * j - g.w_slots, abort_flag);
            if (!__all_sync(0xffffffffu, ok)) break;  // the warp leaves together
            tc_fence_after_sync();
            expand_row(w, a_lane + sw * 32);
            if (pr.both(j)) expand_row(w + 4, a_lane + (sw + 1) * 32);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar0 + 8 * (L::EMPTY_P + static_cast<uint32_t>(j) % PS));
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive_at_leader<CG>(lead_bar0 + 8 * (L::READY + j % L::NE));
            if (j + EXP_GROUPS < pairs) ok = fetch(j + EXP_GROUPS);
            sw += 2 * EXP_GROUPS;
            while (sw >= g.w_slots) sw -= g.w_slots;
        }
        pdl_wait();  // before these warps turn to the epilogue
    }

    if (warp == 3) {
        // One warp polls for the end of the main loop; the epilogue warps sleep in a named barrier until then.  (Twelve
        // polling warps load the path that the mbarrier and TMA instructions of the producers go through: a request then
        // took its thread 370 cycles instead of 50.)
        mbar_wait(bar0 + 8 * L::ACC_FULL, 0, abort_flag);
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (WORKERS + 1)) : "memory");
    } else if (warp >= WORK0 && warp < HELP0) {
        // ------------------------------------------------------------ epilogue: twelve warps
        const int n = n0 + (warp & 3) * 32 + lane;  // this lane's channel
        float comb = 0.f, comb2 = 0.f, bias = 0.f;
        int zterm = 0;  // (128 - zero) * sum of the channel's weight codes
        if (n < p.N) {
            if (p.act_zero) zterm = (128 - __ldg(p.act_zero)) * __ldg(p.w_code_sums + n);
            if (p.w_scale) {
                comb = (p.act_scale ? ld_pinned(p.act_scale) : 0.f) * ld_pinned(p.w_scale + n);
                if (TWO) comb2 = ld_pinned(g.act_scale2) * ld_pinned(p.w_scale + n);
                if (p.bias) bias = __half2float(p.bias[n]);
                if (p.act_zero) bias = fmaf(static_cast<float>(zterm), comb, bias);
                if (p.bos && p.Y && tok0 == 0 && warp < WORK0 + 4)
                    for (int b = 0; b < p.batch; ++b)
                        p.Y[static_cast<long long>(b) * MIXDQ_TOKENS_PER_PROMPT * p.ldy + n] = p.bos_out[n];
            }
        }
        if (W4) {  // the sums carry the factor 16 of the nibble placement: an exact power of two
            comb *= 0.0625f;
            comb2 *= 0.0625f;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (WORKERS + 1)) : "memory");  // (warp 3 has seen the accumulator complete)
        const bool ok = !*abort_flag;
        tc_fence_after_sync();
        const uint32_t acc = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const bool pairs_ok = ((p.N | static_cast<int>(p.ldy)) & 1) == 0 && (reinterpret_cast<uintptr_t>(p.Y) & 3) == 0;
        const int cols = min(g.nt, p.M - tok0);
        if (ok && p.Y && pairs_ok && !p.acc_out) {
            const int who = (warp - WORK0) >> 2;
            __half* col = p.Y + (n & ~1);
            if (cols > 32)
                store_tokens<TWO ? ACC_TWO_BRANCHES : ACC_INT, 16>(acc, acc + g.acc2, 16 * who, 16 * EXP_GROUPS, cols, comb, comb2, bias, col, p.ldy, tok0, p.M, n < p.N,
                                      p.bos != 0, lane);
            else
                store_tokens<TWO ? ACC_TWO_BRANCHES : ACC_INT, 8>(acc, acc + g.acc2, 8 * who, 8 * EXP_GROUPS, cols, comb, comb2, bias, col, p.ldy, tok0, p.M, n < p.N,
                                     p.bos != 0, lane);
        } else if (ok) {
            // odd widths, and the raw sums of the parity hook
            for (int c0 = ((warp - WORK0) >> 2) * 8; c0 < cols; c0 += 8 * EXP_GROUPS) {
                uint32_t r[8], r2[8];
                tmem_ld_32x8(acc + c0, r);
                if (TWO) tmem_ld_32x8(acc + g.acc2 + c0, r2);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    int m = tok0 + c0 + j;
                    if (m >= p.M || n >= p.N) continue;
                    const int32_t a = static_cast<int32_t>(r[j]);
                    float v = fmaf(__int2float_rn(a), comb, bias);
                    if (p.acc_out) p.acc_out[static_cast<long long>(m) * p.N + n] = (W4 ? (a >> 4) : a) + zterm;
                    if (TWO) {
                        const int32_t a2 = static_cast<int32_t>(r2[j]);
                        v = fmaf(__int2float_rn(a2), comb2, v);
                        if (g.acc_out2) g.acc_out2[static_cast<long long>(m) * p.N + n] = W4 ? (a2 >> 4) : a2;
                    }
                    if (p.bos) m += m / (MIXDQ_TOKENS_PER_PROMPT - 1) + 1;
                    if (p.Y) p.Y[m * p.ldy + n] = __float2half_rn(v);
                }
            }
        }
    }

    report_abandoned_wait(abort_flag, p.status);
    tc_fence_before_sync();
    __syncthreads();
    if (CG == 2) cluster_sync();  // neither CTA leaves while its peer may still signal its barriers or use its memory
    if (warp == 0) {
        if (CG == 1)
            tmem_dealloc(tmem_base, 512);
        else
            tmem_dealloc_pair(tmem_base, 512);
    }
}

template <int CG, bool W4, bool TWO>
int launch_t(const CUtensorMap* maps, const TmaParams& tp, ChanArgs g, cudaStream_t stream)
{
    using L = Chan<CG, W4>;
    auto kernel = chan_gemm_kernel<CG, W4, TWO>;
    if (ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), SMEM_MAX) != MIXDQ_OK) return MIXDQ_ERR_CUDA;
    const int x_bytes = g.nt / CG * BK;
    // 12, 8 or 4 activation slots: the pair whose commit frees a slot, and the pair that last used the barrier of the one
    // that will fill it, then belong to the same MMA issuer, so that the barrier's phase is over
    g.x_slots = std::min(L::XS_MAX, (SMEM_MAX - L::OFF_X) / x_bytes) & ~3;
    const int acc_cols = g.nt <= 128 ? (TWO ? 256 : 128) : 256;
    g.acc2 = TWO ? 128 : 0;
    g.w_slots = W4 ? (512 - acc_cols) / 32 : L::WS_MAX;
    g.a_col = acc_cols;
    const int tiles = g.c_tiles * static_cast<int>(ceil_div(tp.M, g.nt));
    return launch_pdl_cluster(kernel, dim3(static_cast<unsigned>(CG * tiles)), dim3(THREADS),
                              static_cast<size_t>(L::OFF_X + g.x_slots * x_bytes), stream, CG, 1u, maps[0], maps[1], maps[2], maps[3],
                              tp, g);
}

template <bool TWO>
int launch(const CUtensorMap* maps, const TmaParams& tp, const ChanArgs& g, int cg, bool w4, cudaStream_t stream)
{
    if (cg == 2) return w4 ? launch_t<2, true, TWO>(maps, tp, g, stream) : launch_t<2, false, TWO>(maps, tp, g, stream);
    return w4 ? launch_t<1, true, TWO>(maps, tp, g, stream) : launch_t<1, false, TWO>(maps, tp, g, stream);
}

}  // namespace

// Tensor maps of one branch: its weights [N, taps * cin] and its activations, int8 [M, cin] or the NHWC image of cin channels
// (with its border when pad is set).  w_rows: channels of a weight tile that arrive, CH but for the self-test.
int encode_chan_branch(CUtensorMap* tw, CUtensorMap* tx, const Params& p, bool conv, int pad, int cin, const void* packed, bool w4, bool wide,
                       const int8_t* codes, int rows, int w_rows)
{
    const int64_t K = (conv ? 9ll : 1ll) * cin;
    const int64_t pitch = row_pitch_bytes(K, w4 ? 4 : 8, MIXDQ_LAYOUT_DEVICE);
    const int rc = w4 ? encode_tmap_2d_u8(tw, packed, static_cast<uint64_t>(pitch), p.N, pitch, wide ? BK : BK / 2, w_rows,
                                          wide ? SWIZZLE_128 : SWIZZLE_64)
                      : encode_tmap_2d_u8(tw, packed, static_cast<uint64_t>(K), p.N, pitch, BK, w_rows, SWIZZLE_128);
    if (rc != MIXDQ_OK) return rc;
    if (conv) return encode_tmap_im2col3x3(tx, codes, false, p.batch, p.H + 2 * pad, p.W + 2 * pad, cin, pad, p.stride, BK, rows);
    return encode_tmap_2d_u8(tx, codes, static_cast<uint64_t>(cin), static_cast<uint64_t>(p.M), static_cast<uint64_t>(cin), BK,
                             static_cast<uint32_t>(rows), SWIZZLE_128);
}

bool chan_tile_ok(int cg, int tokens)
{
    return (cg == 1 || cg == 2) && tokens >= 16 * cg && tokens % (16 * cg) == 0 && tokens <= TOK_MAX && tokens / cg <= ROWS_MAX;
}

// codes: int8 activations, [M, K] rows, or the NHWC image (with its border when p.act_zero).  second: the other branch of a
// shortcut-split layer (p.K or p.Cin, p.act_scale, p.acc_out, packed and codes are then the first branch's).
int run_chan(const Params& p, int amode, const void* packed, int w_bits, const int8_t* codes, int cg, int tokens, cudaStream_t stream,
             const ChanBranch* second)
{
    const bool w4 = w_bits == 4, conv = amode == A_CONV3;
    if (!chan_tile_ok(cg, tokens) || p.addend || (second && tokens > CHAN_TWO_TOKENS)) return MIXDQ_ERR_INVALID_ARG;
    const int pad = (conv && p.act_zero) ? 1 : 0;
    TmaParams tp{};
    tp.M = p.M;
    tp.N = p.N;
    tp.bos = amode == A_BOS;
    tp.batch = p.batch;
    tp.act_scale = p.act_scale;
    tp.act_zero = p.act_zero;
    tp.w_code_sums = p.w_code_sums;
    tp.w_scale = p.w_scale;
    tp.bias = p.bias;
    tp.bos_out = p.bos_out;
    tp.Y = p.Y;
    tp.ldy = p.ldy;
    tp.acc_out = p.acc_out;
    tp.status = p.status;
    const int cin = conv ? p.Cin : p.K, rows = tokens / cg;
    ChanArgs g{};
    g.nt = tokens;
    g.c_tiles = static_cast<int>(ceil_div(p.N, CH * cg));
    // 128 packed bytes of a row are two consecutive k-blocks, unless the channels of a filter tap end inside a k-block
    g.wide = w4 && (!conv || (cin % BK == 0 && (!second || second->cin % BK == 0)));
    tp.cblocks = static_cast<int>(ceil_div(cin, BK));
    tp.k_blocks = (conv ? 9 : 1) * tp.cblocks;
    if (conv) {
        tp.conv = 1;
        tp.pad = pad;
        tp.stride = p.stride;
        tp.Cin = p.Cin;
        tp.HoWo = p.Ho * p.Wo;
        tp.Wo = p.Wo;
    }
    CUtensorMap maps[4]{};  // weights, activations; the second branch's
    // self-test of the bounded waits: half of every weight tile of the last branch never comes, so that the waits on the first
    // of them run out.  (A producer that left tiles out would do for any of them, but a test of it in the kernel, even a bound
    // passed in, cost the 4096 x 640 x 640 W8 layer 0.13 to 0.2 us.)
    const int last_rows = p.test_drop_b_kblock ? CH / 2 : CH;
    int rc = encode_chan_branch(&maps[0], &maps[1], p, conv, pad, cin, packed, w4, g.wide, codes, rows, second ? CH : last_rows);
    if (rc != MIXDQ_OK) return rc;
    if (!second) return launch<false>(maps, tp, g, cg, w4, stream);
    rc = encode_chan_branch(&maps[2], &maps[3], p, conv, pad, second->cin, second->packed, w4, g.wide, second->codes, rows,
                            last_rows);
    if (rc != MIXDQ_OK) return rc;
    g.kb_lo = tp.k_blocks;
    g.cblocks2 = static_cast<int>(ceil_div(second->cin, BK));
    g.Cin2 = conv ? second->cin : 0;
    g.act_scale2 = second->act_scale;
    g.acc_out2 = second->acc_out;
    tp.k_blocks += (conv ? 9 : 1) * g.cblocks2;
    return launch<true>(maps, tp, g, cg, w4, stream);
}

}  // namespace i8
}  // namespace mixdq
