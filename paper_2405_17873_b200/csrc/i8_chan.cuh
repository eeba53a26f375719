// Parts shared by the channel-major int8 kernels (i8_chan.cu: one tile per CTA or CTA pair; i8_chan_many.cu: pairs that walk
// several tiles; wo_chan.cu: fp16 activations).
#pragma once

#include "cta_pair.cuh"
#include "i8_tiles.cuh"

namespace mixdq {
namespace i8 {

constexpr int CH = 128;  // channels of one CTA

// A load that stays where it is written (the compiler moves plain read-only loads down to their first use, past the
// barriers these are meant to overlap).
__device__ __forceinline__ float ld_pinned(const float* p)
{
    float v;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

template <int CG>
__device__ __forceinline__ void arrive_at_leader(uint32_t bar)
{
    if (CG == 1)
        mbar_arrive(bar);
    else
        mbar_arrive_cluster(bar);
}

template <int CG>
__device__ __forceinline__ void commit_mmas(uint32_t bar)
{
    if (CG == 1)
        tc_commit(bar);
    else
        tc_commit_pair(bar, 3);
}

// Where a k-block lies: reduction elements [c * BK, ...) of filter tap `tap` (a linear layer is one endless tap).
struct KPos {
    int tap, c;
    __device__ __forceinline__ KPos(int i, int cblocks) : tap(0), c(i)
    {
        if (i >= cblocks) {  // (not for a linear layer: a division takes 120 cycles of the first request's way)
            tap = i / cblocks;
            c = i - tap * cblocks;
        }
    }
    __device__ __forceinline__ void advance(int n, int cblocks)
    {
        for (c += n; c >= cblocks; c -= cblocks) ++tap;
    }
};

// The k-blocks of a tile as pairs; with two branches each branch's pairs start at its own first k-block.
template <bool TWO>
struct Pairs {
    int nkb, lo, kb_lo, n;  // k-blocks; TWO: pairs and k-blocks of the first branch; pairs in all
    __device__ __forceinline__ Pairs(int nkb_, int kb_lo_)
        : nkb(nkb_), lo(TWO ? (kb_lo_ + 1) >> 1 : 0), kb_lo(kb_lo_), n(TWO ? lo + ((nkb_ - kb_lo_ + 1) >> 1) : (nkb_ + 1) >> 1)
    {
    }
    __device__ __forceinline__ bool second(int j) const { return TWO && j >= lo; }
    __device__ __forceinline__ bool both(int j) const  // whether the pair has two k-blocks
    {
        if (!TWO) return 2 * j + 1 < nkb;
        return j < lo ? 2 * j + 1 < kb_lo : 2 * (j - lo) + 1 < nkb - kb_lo;
    }
};

// A TMA producer, one of two warps that take alternate units, pairs of k-blocks; request(slot, barrier, unit,
// position) asks for one.  A warp that runs alone takes some five cycles per instruction, so a
// loop over k-blocks costs 370 cycles a turn whatever the size of the request, and an integer division in it 120 more.
// Hence the two warps and the running position, and the first lap of the ring, which waits for nothing, goes out from all
// lanes of the first of them at once (65 cycles apart).  free[unit % barriers] says that the slot of the unit `slots`
// positions later is free; `barriers` is even and at least `slots`: a warp meets every phase.
template <bool TWO, typename F>
__device__ __forceinline__ void produce(int which, int lane, int slots, const Pairs<TWO>& pr, int cblocks, int cblocks2, uint32_t free,
                                        int barriers, volatile int* abort_flag, F&& request)
{
    const int units = pr.n;
    if (which == 0 && lane < slots && lane < units)
        request(lane, lane, lane, pr.second(lane) ? KPos(2 * (lane - pr.lo), cblocks2) : KPos(2 * lane, cblocks));
    __syncwarp();
    if (slots + which >= units) return;
    int s = which, q = which, sb = which + slots;
    if (s >= slots) s -= slots;
    if (sb >= barriers) sb -= barriers;
    uint32_t par = 0;
    KPos at(2 * (slots + which), cblocks);
    bool second = false;
    for (int i = slots + which; i < units; i += 2) {
        if (TWO && !second && pr.second(i)) {
            second = true;
            cblocks = cblocks2;
            at = KPos(2 * (i - pr.lo), cblocks2);
        }
        const bool ok = mbar_wait(free + 8 * q, par, abort_flag);
        if (!__all_sync(0xffffffffu, ok)) break;
        if (elect_one()) request(s, sb, i, at);
        __syncwarp();
        at.advance(4, cblocks);
        s += 2;
        while (s >= slots) s -= slots;
        sb += 2;
        if (sb >= barriers) sb -= barriers;
        q += 2;
        if (q >= barriers) {
            q -= barriers;
            par ^= 1;
        }
    }
}

// The packed int4 rows of a pair of k-blocks as they lie in shared memory: 128-byte rows (both k-blocks of a channel, 128-byte
// swizzle) where the pair is contiguous in memory, else two tiles of 64-byte rows (64-byte swizzle).  The swizzle makes the
// reads of a warp, a row per lane, conflict-free.
struct PackedRows {
    uint32_t row_ofs, swz;
    bool wide;
    __device__ __forceinline__ PackedRows(int row, bool wide_)
        : row_ofs(row * (wide_ ? 128u : 64u)), swz((static_cast<uint32_t>(wide_ ? row : (row >> 1) & 3) & 7u) << 4), wide(wide_)
    {
    }
    __device__ __forceinline__ void load(const uint8_t* slot, uint4 (&w)[8]) const
    {
        const uint8_t* src = slot + row_ofs;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            // (wide: the second k-block is chunks 4 .. 7 of the row, and the swizzle runs over all eight)
            const uint32_t ofs = static_cast<uint32_t>(k & 3) << 4;
            w[k] = *reinterpret_cast<const uint4*>(src + (k < 4 ? ofs ^ swz : (wide ? (ofs | 64u) ^ swz : (ofs ^ swz) + CH * BK / 2)));
        }
    }
};

// 64 packed bytes of a channel -> its 32 tensor-memory columns of int8 codes (times 16: a nibble in the high half of a byte).
__device__ __forceinline__ void expand_row(const uint4* w, uint32_t taddr)
{
    uint32_t c[32];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t v[4] = {w[k].x, w[k].y, w[k].z, w[k].w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            c[8 * k + 2 * q] = (v[q] << 4) & 0xF0F0F0F0u;
            c[8 * k + 2 * q + 1] = v[q] & 0xF0F0F0F0u;
        }
    }
    tmem_st_32x32(taddr, c);
}

// G consecutive columns of this warp's 32 lanes.
template <int G>
__device__ __forceinline__ void tmem_ld_tokens(uint32_t taddr, uint32_t (&r)[G])
{
    static_assert(G == 8 || G == 16, "");
    if constexpr (G == 8)
        tmem_ld_32x8(taddr, r);
    else
        tmem_ld_32x16(taddr, r);
}

// One warp's share of the epilogue: its 32 lanes' channels x the groups of G tokens at c0, c0 + step, ...  Lanes 2 i and 2 i + 1
// swap halves of a packed token pair and each stores both channels of one token: a store covers 64 contiguous bytes of two
// output rows.  col: Y at the lane's channel pair.  A turn is bound by its latencies (tensor-memory load, conversions, swap):
// sixteen tokens a turn where there are enough of them.
enum : int {
    ACC_INT = 0,           // y = acc * comb + bias
    ACC_TWO_BRANCHES = 1,  // y = acc2 * comb2 + (acc * comb + bias)
    ACC_FLOAT = 2,         // fp32 sums in two accumulators: y = (acc + acc2) * comb + bias
};
template <int KIND, int G>
__device__ __forceinline__ void store_tokens(uint32_t acc, uint32_t acc2, int c0, int step, int cols, float comb, float comb2, float bias,
                                             __half* col, long long ldy, int tok0, int M, bool in_n, bool bos, int lane)
{
    const uint32_t sel = (lane & 1) ? 0x3276u : 0x5410u;  // odd: token 1 (other's, own); even: token 0 (own, other's)
    const bool all_n = __all_sync(0xffffffffu, in_n);
    for (; c0 < cols; c0 += step) {
        uint32_t r[G], r2[G], own[G / 2];
        tmem_ld_tokens<G>(acc + c0, r);
        if (KIND != ACC_INT) tmem_ld_tokens<G>(acc2 + c0, r2);
        tmem_ld_wait();
        const int m0 = tok0 + c0 + (lane & 1);
#pragma unroll
        for (int j = 0; j < G / 2; ++j) {
            float a, b;
            if (KIND == ACC_FLOAT) {
                a = fmaf(__uint_as_float(r[2 * j]) + __uint_as_float(r2[2 * j]), comb, bias);
                b = fmaf(__uint_as_float(r[2 * j + 1]) + __uint_as_float(r2[2 * j + 1]), comb, bias);
            } else {
                a = fmaf(__int2float_rn(static_cast<int32_t>(r[2 * j])), comb, bias);
                b = fmaf(__int2float_rn(static_cast<int32_t>(r[2 * j + 1])), comb, bias);
            }
            if (KIND == ACC_TWO_BRANCHES) {
                a = fmaf(__int2float_rn(static_cast<int32_t>(r2[2 * j])), comb2, a);
                b = fmaf(__int2float_rn(static_cast<int32_t>(r2[2 * j + 1])), comb2, b);
            }
            const __half2 h = __floats2half2_rn(a, b);
            own[j] = *reinterpret_cast<const uint32_t*>(&h);
        }
#pragma unroll
        for (int j = 0; j < G / 2; ++j) own[j] = __byte_perm(own[j], __shfl_xor_sync(0xffffffffu, own[j], 1), sel);
        __half* dst = col + m0 * ldy;
        if (all_n && !bos && c0 + G <= cols) {  // (uniform: the whole group of tokens exists)
#pragma unroll
            for (int j = 0; j < G / 2; ++j) *reinterpret_cast<uint32_t*>(dst + 2 * j * ldy) = own[j];
        } else if (in_n) {
#pragma unroll
            for (int j = 0; j < G / 2; ++j) {
                int m = m0 + 2 * j;
                if (m >= M || c0 + 2 * j + (lane & 1) >= cols) continue;
                if (bos) m += m / (MIXDQ_TOKENS_PER_PROMPT - 1) + 1;
                *reinterpret_cast<uint32_t*>(col + m * ldy) = own[j];
            }
        }
    }
}

int encode_chan_branch(CUtensorMap* tw, CUtensorMap* tx, const Params& p, bool conv, int pad, int cin, const void* packed, bool w4,
                       bool wide, const int8_t* codes, int rows, int w_rows = CH);

}  // namespace i8
}  // namespace mixdq
