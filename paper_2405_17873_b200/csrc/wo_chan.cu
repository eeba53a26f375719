// Weight-only (W2 / W3 / W4 / W8, fp16 activations) layers of one wave, channel-major: the weights on the 128 rows of the
// tensor-core tile, expanded to fp16 (code - zero, exact integers) straight into tensor memory, the tokens on its N side.
//
// Why.  The two-CTA form with the tokens on the rows (i8_pair.cu, MODE 3) writes every expanded weight row to shared memory
// and reads it back, its tiles of 256 rows leave SMs idle, and its expansion bounds the main loop.  Here a packed row goes
// through shared memory once, a tile has any multiple of 16 tokens, and expansion runs ahead of the previous kernel: the
// weights are constants of the layer.  See i8_chan.cu for the pipeline, which is the same but for three things:
//   * a pair of k-blocks is 2 x 64 elements: one packed block of 128 codes;
//   * fp32 sums depend on their order, so each MMA issuer has an accumulator of its own and the epilogue adds the two:
//     results do not change from run to run;
//   * there is no quantization pass: the activations are the layer's input as it is.
//
// Measured on B200, before and now: W4 16 x 10240 x 1280 7.4 -> 5.0 us, 17 x 1280 x 1280 10.2 -> 4.2, 128 x 1280 x 5120 38.4 ->
// 13.5, 256 x 1280 x 1280 8.4 -> 5.2, 1024 x 1280 x 1280 10.1 -> 6.3, 1024 x 1280 x 5120 23.7 -> 15.2, 3x3 convolution 48 x 48
// x 640 -> 640 28.9 -> 17.6; W3 the first two 7.5 -> 5.2, 10.4 -> 4.3; W8 16 x 10240 x 1280 7.4 -> 5.0, 17 x 1280 x 1280 10.2
// -> 4.1, 1024 x 1280 x 1280 10.9 -> 6.4, 1024 x 1280 x 5120 25.0 -> 15.  A long reduction takes 300 cycles per k-block of 64:
// the expansion (three groups of four warps, some 1700 cycles for a pair of k-blocks; 3 bits more) and the rings' latency.
#include <algorithm>

#include "i8_chan.cuh"

namespace mixdq {
namespace wo {

namespace {

using namespace i8;

constexpr int BKE = 64;        // fp16 elements of a k-block (128-byte rows)
constexpr int EXP_GROUPS = 3;  // of four warps: expansion, then epilogue
constexpr int WORKERS = 4 * EXP_GROUPS, WORK0 = 4, HELP0 = WORK0 + WORKERS;
constexpr int THREADS = (HELP0 + 2) * 32;
constexpr int SMEM_MAX = 232448;
constexpr int TOK_MAX = 192;   // two accumulators and two pairs of expanded weights fill tensor memory
// Warps: 0 and 3 MMA issuers (leader), 1 and 16 weight producers, 2 and 17 activation producers, 4 .. 15 expansion, then
// epilogue.
constexpr int NE = 6;          // pairs whose barriers exist at a time: at least the deepest ring
constexpr int PS = 6;          // packed slots, a pair each
constexpr int READY = 0;       // leader: token rows and expanded weights of both CTAs are in place
constexpr int EMPTY = READY + NE;
constexpr int FULL_P = EMPTY + NE;
constexpr int EMPTY_P = FULL_P + PS;
constexpr int ACC_FULL = EMPTY_P + PS;
constexpr int NUM_BARS = ACC_FULL + 1;
constexpr int OFF_MISC = NUM_BARS * 8;
constexpr int OFF_P = 1024;
static_assert(OFF_MISC + 16 <= OFF_P && NE % EXP_GROUPS == 0 && PS % EXP_GROUPS == 0 && NE % 2 == 0,
              "layout; a waiter must meet every phase of the barriers it waits on");

template <int BITS>
constexpr int kPackedBytes = CH * 16 * BITS;  // of a pair's rows
template <int BITS>
constexpr int kXOffset = OFF_P + PS * kPackedBytes<BITS>;

struct WoArgs {
    int nt;        // tokens of a tile (multiple of 16 CG)
    int c_tiles;   // channel tiles (128 CG channels each)
    int x_slots, w_slots;
    int acc2;      // column of the second accumulator
    const int32_t* w_zero;  // nullptr: signed codes
};

// A row's packed block of 128 codes in registers: 4 bits 16 words (byte i of a word = code i | code i + 4 << 4), 2 and 3 bits
// four words per bit plane.
template <int BITS>
struct Codes {
    uint4 v[BITS];
    __device__ __forceinline__ void load(const uint8_t* slot, int row)
    {
        // 64-byte rows come with the 64-byte swizzle; rows of 48 bytes are conflict-free, of 32 two-way, as they are
        // (8 bits: 128-byte rows, 128-byte swizzle)
        const uint32_t swz = BITS == 8 ? (static_cast<uint32_t>(row) & 7u) << 4 : (BITS == 4 ? (static_cast<uint32_t>(row >> 1) & 3u) << 4 : 0u);
        const uint8_t* src = slot + row * (16 * BITS);
#pragma unroll
        for (int k = 0; k < BITS; ++k) v[k] = *reinterpret_cast<const uint4*>(src + ((static_cast<uint32_t>(k) << 4) ^ swz));
    }
    static __device__ __forceinline__ uint32_t word(const uint4& q, int i)
    {
        return i == 0 ? q.x : (i == 1 ? q.y : (i == 2 ? q.z : q.w));
    }
    // Eight codes of group j of k-block h as nibbles of a word (not for 8 bits).
    __device__ __forceinline__ uint32_t group(int h, int j, uint32_t flip) const
    {
        if constexpr (BITS == 4) {
            return word(v[2 * h + (j >> 2)], j & 3) ^ flip;
        } else {
            uint32_t w = 0;
#pragma unroll
            for (int b = 0; b < BITS; ++b) w |= ((word(v[b], 2 * h + (j >> 2)) >> (j & 3)) & 0x11111111u) << b;
            return w;
        }
    }
};

// 64 codes -> 32 tensor-memory columns of fp16 pairs.  1024 + u has the fp16 bits 0x6400 | u for an integer u < 1024, so the
// difference (1024 + u) - (1024 + zero) is exact.
template <int BITS>
__device__ __forceinline__ void expand_codes(const Codes<BITS>& codes, int h, uint32_t flip, __half2 z2, uint32_t taddr)
{
    uint32_t c[32];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        uint32_t lo4, hi4;  // codes 0 .. 3 and 4 .. 7 of the group as bytes
        if constexpr (BITS == 8) {
            const uint4& v = codes.v[4 * h + (j >> 1)];
            lo4 = ((j & 1) ? v.z : v.x) ^ flip;
            hi4 = ((j & 1) ? v.w : v.y) ^ flip;
        } else {
            const uint32_t w = codes.group(h, j, flip);
            lo4 = w & 0x0F0F0F0Fu;
            hi4 = (w >> 4) & 0x0F0F0F0Fu;
        }
        const uint32_t b[4] = {__byte_perm(lo4, 0x64646464u, 0x5140), __byte_perm(lo4, 0x64646464u, 0x7362),
                               __byte_perm(hi4, 0x64646464u, 0x5140), __byte_perm(hi4, 0x64646464u, 0x7362)};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&b[q]), z2);
            c[4 * j + q] = *reinterpret_cast<const uint32_t*>(&d);
        }
    }
    tmem_st_32x32(taddr, c);
}

// Grid: CG CTAs (a cluster) per tile of 128 CG channels x nt tokens, channel tiles fastest.
template <int CG, int BITS>
__global__ void __launch_bounds__(THREADS, 1)
wo_chan_kernel(const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ CUtensorMap tmap_x, const TmaParams p, const WoArgs g)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + OFF_MISC);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + OFF_MISC + 4);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
    const bool leader = rank == 0;
    const int tile = static_cast<int>(blockIdx.x) / CG;
    const Pairs<false> pr(p.k_blocks, 0);
    const int pairs = pr.n, rows = g.nt / CG;  // token rows this CTA holds
    const int tok0 = (tile / g.c_tiles) * g.nt;
    const int n0 = (tile % g.c_tiles) * (CG * CH) + static_cast<int>(rank) * CH;
    const uint32_t x_bytes = static_cast<uint32_t>(rows) * 2 * BKE;
    constexpr int P_BYTES = kPackedBytes<BITS>;

    const uint32_t bar0 = smem_u32(smem), p0 = bar0 + OFF_P, x0 = bar0 + kXOffset<BITS>;
    const uint32_t lead_bar0 = CG == 2 ? map_to_cta(bar0, 0) : bar0;

    pdl_launch_dependents();
    if (warp == 3 && lane == 0) {
        for (int s = 0; s < NE; ++s) {
            mbar_init(bar0 + 8 * (READY + s), 1 + CG * 4);  // activation bytes; a group's four warps of each CTA
            mbar_init(bar0 + 8 * (EMPTY + s), 1);
        }
        for (int s = 0; s < PS; ++s) {
            mbar_init(bar0 + 8 * (FULL_P + s), 1);
            mbar_init(bar0 + 8 * (EMPTY_P + s), 4);
        }
        mbar_init(bar0 + 8 * ACC_FULL, 2);  // one commit of each issuer
        *abort_flag = (smem_u32(smem) & 1023u) ? 1 : 0;
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
    constexpr uint32_t tmem_base = 0;  // all 512 columns are this CTA's
    if (*s_tmem != tmem_base) *abort_flag = 1;
    const int a_col = 2 * g.acc2;
    // the weights are constants of the layer: their producers and the warps that expand them run ahead of earlier kernels
    const bool expander = warp >= WORK0 && warp < HELP0;
    if (warp != 1 && warp != HELP0 && !expander) pdl_wait();

    if (warp == 0 || warp == 3) {
        // ------------------------------------------------------------ MMA issuers (two warps of the leader), alternate pairs
        if (leader) {
            const uint32_t idesc = make_idesc(1, 0, CG * CH, static_cast<uint32_t>(g.nt));
            const uint64_t x_desc0 = smem_desc_sw128(x0);
            const int first = warp == 0 ? 0 : 1;
            const uint32_t acc = tmem_base + first * g.acc2;
            int sx = 2 * first % g.x_slots, sw = 2 * first % g.w_slots, sb = first;
            uint32_t par = 0;
            for (int j = first; j < pairs; j += 2) {
                const bool ok = mbar_wait(bar0 + 8 * (READY + sb), par, abort_flag);
                if (!__all_sync(0xffffffffu, ok)) break;
                tc_fence_after_sync();
                const uint64_t x_desc = x_desc0 + static_cast<uint32_t>(sx) * (x_bytes >> 4);
                const uint32_t a = tmem_base + a_col + sw * 32;
                const bool both = pr.both(j);
                if (elect_one()) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (h == 1 && !both) break;
                        const uint64_t xd = x_desc + h * (x_bytes >> 4);
#pragma unroll
                        for (int k = 0; k < BKE / 16; ++k)
                            mma_f16_ts<CG>(acc, a + 32 * h + 8 * k, xd + 2 * k, idesc, (j != first || h != 0 || k != 0) ? 1u : 0u);
                    }
                    commit_mmas<CG>(bar0 + 8 * (EMPTY + sb));
                    if (j + 2 >= pairs) commit_mmas<CG>(bar0 + 8 * ACC_FULL);
                }
                __syncwarp();
                sx += 4;
                while (sx >= g.x_slots) sx -= g.x_slots;
                sw += 4;
                while (sw >= g.w_slots) sw -= g.w_slots;
                sb += 2;
                if (sb >= NE) {
                    sb -= NE;
                    par ^= 1;
                }
            }
            if (first >= pairs && elect_one()) commit_mmas<CG>(bar0 + 8 * ACC_FULL);  // (nothing to wait for)
            __syncwarp();
        }
    } else if (warp == 1 || warp == HELP0) {
        // ------------------------------------------------------------ packed weight rows of this CTA's channels
        auto request = [&](int s, int, int u, KPos) {
            const uint32_t full = bar0 + 8 * (FULL_P + s);
            mbar_arrive_expect_tx(full, P_BYTES);
            tma_load_2d(p0 + s * P_BYTES, &tmap_w, u * 16 * BITS, n0, full);
        };
        Pairs<false> requested = pr;
        if (p.test_drop_b_kblock) requested.n = min(pr.n, p.test_drop_b_kblock - 1);
        produce<false>(warp == 1 ? 0 : 1, lane, PS, requested, 1 << 30, 1, bar0 + 8 * EMPTY_P, PS, abort_flag, request);
    } else if (warp == 2 || warp == HELP0 + 1) {
        // ------------------------------------------------------------ fp16 token rows by TMA
        const int m0 = tok0 + static_cast<int>(rank) * rows;
        int img = 0, wi = 0, hi = 0;
        if (p.conv) {
            const int mc = m0 < p.M ? m0 : 0;  // no output rows: any pixels will do
            img = mc / p.HoWo;
            const int rem = mc - img * p.HoWo;
            const int ho = rem / p.Wo;
            hi = p.stride * ho - 1;
            wi = p.stride * (rem - ho * p.Wo) - 1;
        }
        auto request = [&](int s, int sb, int u, KPos at) {
            const uint32_t full = bar0 + 8 * (READY + sb), lead_full = lead_bar0 + 8 * (READY + sb);
            const int n = pr.both(u) ? 2 : 1;
            if (leader) mbar_arrive_expect_tx(full, n * CG * x_bytes);
            for (int h = 0; h < n; ++h) {
                const uint32_t dst = x0 + (2 * s + h) * x_bytes;
                if (p.conv) {
                    const int kh = at.tap / 3, kw = at.tap - 3 * kh;
                    if (CG == 1)
                        tma_load_im2col(dst, &tmap_x, at.c * BKE, wi, hi, img, kw, kh, full);
                    else
                        tma_load_im2col_pair(dst, &tmap_x, at.c * BKE, wi, hi, img, kw, kh, lead_full);
                } else if (CG == 1) {
                    tma_load_2d(dst, &tmap_x, at.c * BKE, m0, full);
                } else {
                    tma_load_2d_pair(dst, &tmap_x, at.c * BKE, m0, lead_full);
                }
                at.advance(1, p.cblocks);
            }
        };
        produce<false>(warp == 2 ? 0 : 1, lane, g.x_slots / 2, pr, p.cblocks, 1, bar0 + 8 * EMPTY, NE, abort_flag, request);
    } else if (expander) {
        // ------------------------------------------------------------ packed codes -> fp16 in tensor memory
        // A thread owns a channel; groups of four warps take alternate pairs and fetch the next packed rows into registers
        // before they wait for its slots.
        const int group = (warp - WORK0) >> 2, row = (warp & 3) * 32 + lane;
        const uint32_t a_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16) + a_col;
        const uint32_t flip = g.w_zero ? 0u : (BITS == 8 ? 0x80808080u : 0x88888888u);  // signed codes + 128 or 8
        const int zero = g.w_zero ? (n0 + row < p.N ? __ldg(g.w_zero + n0 + row) : 0) : (BITS == 8 ? 128 : 8);
        const __half2 z2 = __half2half2(__int2half_rn(1024 + zero));
        int sw = 2 * group % g.w_slots;  // slot of the pair's first k-block
        Codes<BITS> codes;
        auto fetch = [&](int j) {
            const uint32_t q = static_cast<uint32_t>(j), sp = q % PS;
            const bool ok = mbar_wait(bar0 + 8 * (FULL_P + sp), (q / PS) & 1, abort_flag);
            codes.load(smem + OFF_P + sp * P_BYTES, row);
            return ok;
        };
        bool ok = group < pairs ? fetch(group) : true;
        for (int j = group; j < pairs; j += EXP_GROUPS) {
            if (ok && 2 * j >= g.w_slots) {
                const uint32_t q = static_cast<uint32_t>(2 * j - g.w_slots) >> 1;
                ok = mbar_wait(bar0 + 8 * (EMPTY + q % NE), (q / NE) & 1, abort_flag);
            }
            if (!__all_sync(0xffffffffu, ok)) break;  // the warp leaves together
            tc_fence_after_sync();
            expand_codes<BITS>(codes, 0, flip, z2, a_lane + sw * 32);
            if (pr.both(j)) expand_codes<BITS>(codes, 1, flip, z2, a_lane + (sw + 1) * 32);
            __syncwarp();
            if (lane == 0) mbar_arrive(bar0 + 8 * (EMPTY_P + static_cast<uint32_t>(j) % PS));
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) arrive_at_leader<CG>(lead_bar0 + 8 * (READY + j % NE));
            if (j + EXP_GROUPS < pairs) ok = fetch(j + EXP_GROUPS);
            sw += 2 * EXP_GROUPS;
            while (sw >= g.w_slots) sw -= g.w_slots;
        }
        pdl_wait();  // before these warps turn to the epilogue
    }

    if (warp == 3) {
        // one warp polls for the end of the main loop; the epilogue warps sleep in a named barrier until then
        mbar_wait(bar0 + 8 * ACC_FULL, 0, abort_flag);
        __syncwarp();
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (WORKERS + 1)) : "memory");
    } else if (expander) {
        // ------------------------------------------------------------ epilogue: twelve warps
        const int n = n0 + (warp & 3) * 32 + lane;  // this lane's channel
        float comb = 0.f, bias = 0.f;
        if (n < p.N) {
            comb = ld_pinned(p.w_scale + n);
            if (p.bias) bias = __half2float(p.bias[n]);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * (WORKERS + 1)) : "memory");  // (warp 3 has seen the accumulators complete)
        const bool ok = !*abort_flag;
        tc_fence_after_sync();
        const uint32_t acc = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
        const bool one = pairs == 1;  // the second accumulator was never written
        const bool pairs_ok = ((p.N | static_cast<int>(p.ldy)) & 1) == 0 && (reinterpret_cast<uintptr_t>(p.Y) & 3) == 0;
        const int cols = min(g.nt, p.M - tok0), who = (warp - WORK0) >> 2;
        if (ok && pairs_ok && !one) {
            __half* col = p.Y + (n & ~1);
            if (cols > 32)
                store_tokens<ACC_FLOAT, 16>(acc, acc + g.acc2, 16 * who, 16 * EXP_GROUPS, cols, comb, 0.f, bias, col, p.ldy, tok0, p.M,
                                            n < p.N, false, lane);
            else
                store_tokens<ACC_FLOAT, 8>(acc, acc + g.acc2, 8 * who, 8 * EXP_GROUPS, cols, comb, 0.f, bias, col, p.ldy, tok0, p.M,
                                           n < p.N, false, lane);
        } else if (ok) {
            // odd widths, and reductions of one pair
            for (int c0 = 8 * who; c0 < cols; c0 += 8 * EXP_GROUPS) {
                uint32_t r[8], r2[8];
                tmem_ld_32x8(acc + c0, r);
                tmem_ld_32x8(acc + g.acc2 + c0, r2);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int m = tok0 + c0 + j;
                    if (m >= p.M || n >= p.N) continue;
                    const float sum = __uint_as_float(r[j]) + (one ? 0.f : __uint_as_float(r2[j]));
                    p.Y[m * p.ldy + n] = __float2half_rn(fmaf(sum, comb, bias));
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

template <int CG, int BITS>
int launch_t(const CUtensorMap& tw, const CUtensorMap& tx, const TmaParams& tp, WoArgs g, cudaStream_t stream)
{
    auto kernel = wo_chan_kernel<CG, BITS>;
    if (ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), SMEM_MAX) != MIXDQ_OK) return MIXDQ_ERR_CUDA;
    const int x_bytes = g.nt / CG * 2 * BKE;
    // 12, 8 or 4 activation slots (see launch_t of i8_chan.cu)
    g.x_slots = std::min(2 * NE, (SMEM_MAX - kXOffset<BITS>) / x_bytes) & ~3;
    g.acc2 = g.nt <= 64 ? 64 : (g.nt <= 128 ? 128 : 192);
    g.w_slots = std::min(2 * NE, (512 - 2 * g.acc2) / 32);
    const int tiles = g.c_tiles * static_cast<int>(ceil_div(tp.M, g.nt));
    return launch_pdl_cluster(kernel, dim3(static_cast<unsigned>(CG * tiles)), dim3(THREADS),
                              static_cast<size_t>(kXOffset<BITS> + g.x_slots * x_bytes), stream, CG, 1u, tw, tx, tp, g);
}

template <int BITS>
int launch(int cg, const CUtensorMap& tw, const CUtensorMap& tx, const TmaParams& tp, const WoArgs& g, cudaStream_t stream)
{
    return cg == 2 ? launch_t<2, BITS>(tw, tx, tp, g, stream) : launch_t<1, BITS>(tw, tx, tp, g, stream);
}

}  // namespace

bool chan_tile_ok(int cg, int tokens)
{
    return (cg == 1 || cg == 2) && tokens >= 16 * cg && tokens % (16 * cg) == 0 && tokens <= TOK_MAX && tokens / cg <= 128;
}

// A k-block of a convolution must be a whole block of the flattened reduction index: Cin a multiple of 64.
bool chan_path_ok(const Params& p, int amode, const void* packed, int w_bits)
{
    if ((w_bits <= 3 && !p.w_zero) || !p.Y) return false;
    if (((reinterpret_cast<uintptr_t>(p.X) | reinterpret_cast<uintptr_t>(packed)) & 15) != 0) return false;
    if (amode == A_CONV3) return p.Cin % BKE == 0 && (p.stride == 1 || p.stride == 2);
    return amode == A_LINEAR && p.K % 8 == 0 && p.ldx % 8 == 0;
}

// Cycles of a tile, fitted to 120 layers of 1 to 4096 rows (graphs of launches; error 5 to 7 per cent): fixed part + k-blocks x
// (issue, little of it per token) + epilogue, and the share of the SMs in use (they compete for the L2).  The other forms' as
// fitted to the same layers:
//   * up to 16 rows, a linear layer: the kernels of wo_gemm.cu, which split the reduction inside a CTA and win wherever it is
//     long or the rows are eight at most and the weights few (16 x 1280 x 5120 W4 5.6 us against 13.0), and lose by up to half
//     on many channels (16 x 10240 x 1280 7.4 and 5.0);
//   * 17 to 255 rows: nothing comes near (17 x 1280 x 1280 W4 10.2 us and 4.2, 128 x 1280 x 5120 38 and 13.7), so tiles of
//     more than one wave are taken too;
//   * from 256 rows, with a workspace: the pair form, whose split reductions win on the longest.
int plan_chan(const Params& p, int amode, int w_bits, bool pair, int num_sms, int* cg)
{
    const bool conv = amode == A_CONV3;
    const int k_blocks = static_cast<int>(conv ? 9 * ceil_div(p.Cin, BKE) : ceil_div(p.K, BKE));
    const double nkb = k_blocks;
    double best = 0;
    int tokens = 0;
    for (int c = 1; c <= 2; ++c) {
        const int64_t c_tiles = ceil_div(p.N, CH * c);
        for (int t = 16 * c; chan_tile_ok(c, t) && t < p.M + 16 * c; t += 16 * c) {
            const int64_t ctas = c * c_tiles * ceil_div(p.M, t);
            if (ctas > num_sms && p.M >= 256) continue;
            const double waves = static_cast<double>(ceil_div(ctas, num_sms)), busy = std::min(1.0, static_cast<double>(ctas) / num_sms);
            const double per_kb = (w_bits == 4 ? 244.0 : 284.0) - (c == 2 ? 16.0 : 0.0) + 0.3 * t;
            const double cost = (c == 1 ? 2600.0 : 2900.0) +
                                waves * (nkb * (per_kb + (c == 1 ? 47.0 : 57.0) * busy) + 27.0 * t + (c == 1 ? 2100.0 : 3650.0) * busy);
            if (tokens == 0 || cost < best) {
                best = cost;
                tokens = t;
                *cg = c;
            }
        }
    }
    if (tokens == 0) return 0;
    const double N = p.N, K = p.K, b = w_bits == 4 ? 0.0 : 1.0;
    if (p.M <= 16 && !conv && p.K <= 5120) {
        const double other = p.M <= 8 ? 3950.0 + 220.0 * b + 0.29 * K + (w_bits == 8 ? 3.4e-4 : 4.8e-4 + 1.1e-4 * b) * N * K
                                      : 5560.0 + 0.13 * N + (0.1 + 0.09 * b) * K + 7e-4 * N * K;
        return best < 0.97 * other ? tokens : 0;
    }
    if (pair) return best < pair_cost(p.M, p.N, p.K, k_blocks, w_bits, num_sms) ? tokens : 0;
    return tokens;
}

int run_chan(const Params& p, int amode, const void* packed, int w_bits, int cg, int tokens, cudaStream_t stream)
{
    const bool conv = amode == A_CONV3;
    if (!chan_tile_ok(cg, tokens)) return MIXDQ_ERR_INVALID_ARG;
    TmaParams tp{};
    tp.M = p.M;
    tp.N = p.N;
    tp.w_scale = p.w_scale;
    tp.bias = p.bias;
    tp.Y = p.Y;
    tp.ldy = p.ldy;
    tp.status = p.status;
    tp.test_drop_b_kblock = p.test_drop_b_kblock;
    tp.cblocks = static_cast<int>(ceil_div(conv ? p.Cin : p.K, BKE));
    tp.k_blocks = (conv ? 9 : 1) * tp.cblocks;
    const int rows = tokens / cg;
    CUtensorMap tw, tx;
    int rc;
    if (conv) {
        tp.conv = 1;
        tp.stride = p.stride;
        tp.HoWo = p.Ho * p.Wo;
        tp.Wo = p.Wo;
        rc = encode_tmap_im2col3x3(&tx, p.X, true, p.batch, p.H, p.W, p.Cin, 0, p.stride, BKE, rows);
    } else {
        rc = encode_tmap_2d_f16(&tx, p.X, static_cast<uint64_t>(p.K), static_cast<uint64_t>(p.M), static_cast<uint64_t>(p.ldx), BKE,
                                static_cast<uint32_t>(rows));
    }
    if (rc != MIXDQ_OK) return rc;
    const int64_t pitch = row_pitch_bytes(p.K, w_bits, MIXDQ_LAYOUT_DEVICE);
    rc = encode_tmap_2d_u8(&tw, packed, static_cast<uint64_t>(pitch), static_cast<uint64_t>(p.N), static_cast<uint64_t>(pitch),
                           static_cast<uint32_t>(16 * w_bits), CH, w_bits == 8 ? SWIZZLE_128 : (w_bits == 4 ? SWIZZLE_64 : SWIZZLE_NONE));
    if (rc != MIXDQ_OK) return rc;
    WoArgs g{};
    g.nt = tokens;
    g.c_tiles = static_cast<int>(ceil_div(p.N, CH * cg));
    g.w_zero = p.w_zero;
    if (w_bits == 8) return launch<8>(cg, tw, tx, tp, g, stream);
    if (w_bits == 4) return launch<4>(cg, tw, tx, tp, g, stream);
    if (w_bits == 3) return launch<3>(cg, tw, tx, tp, g, stream);
    return launch<2>(cg, tw, tx, tp, g, stream);
}

}  // namespace wo
}  // namespace mixdq
