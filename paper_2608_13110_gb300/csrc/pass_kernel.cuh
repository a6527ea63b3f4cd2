// Fused staircase pass over the temporal boundary (arXiv 2608.13110,
// Sec. 3.1, Algorithm 1: every paired step contracts two row tensors into the
// boundary). As in the paper's production code (Sec. 5.2), where several small
// tensors are combined first so that the big boundary is touched less often,
// every step of one window of address bits is applied in a single read + write
// of the boundary.
//
// A pass applies a compile-time sequence of controlled 2x2 steps to tiles of
// 2^13 complex64 entries: the window's M address bits in chunks that the
// copies want (see pass_chunk_log2). Chunks that are exactly zero are not
// visited (TileSkip). At a row turn the four steps on the window's two
// outermost bits run as one 4x4 block (composed on the host, see tb_internal.h).
//
// Warp-specialised, one persistent CTA per SM:
//   * one producer warp moves whole tiles between HBM and a 3-stage ring of
//     shared-memory stages with tensor copies (cp.async.bulk.tensor, one per
//     chunk, 128-byte swizzle; 64-byte rows and swizzle for 10-bit windows
//     above bit 0): a load completes on the stage's "full" mbarrier; once the
//     consumers have written the stage back it is stored in place, and as soon
//     as the stores have read the stage the next tile's loads are issued into it;
//   * 8 consumer warps read global memory only for a bitstring's state, a tile
//     ahead, and never wait for one another: warp w owns the 1024 entries of the
//     tile that share 3 "warp bits" and holds them as 32 entries per thread: 5
//     address bits in registers, 5 on the lanes. Every window bit is one of
//     these 10, so a step on a register bit is register arithmetic and a step on
//     a lane bit exchanges the partner lane's entries with warp shuffles. A warp
//     reads its entries from the stage once, applies every step, writes them
//     back and arrives on the stage's "done" mbarrier. HBM traffic, shared-memory
//     traffic and the arithmetic of different warps all overlap.
// The tensor map orders the tile's address bits so that every warp access to
// a stage is free of shared-memory bank conflicts, except in the 64-byte-row
// layout of 10-bit windows, where they are two-way (see slot_of).
//
// What bounds it: HBM and the FP32 pipe about equally. The consumer loop alone
// (no copies) takes, in cycles per tile, 5620 for a 9-bit forward window, 6100
// reversed, 7320 for a 7-bit top turn and 13120 for a 10-bit bottom turn; the
// measured HBM copy rate allows a tile every 6050. A paired FMA whose three
// operands are all fresh registers takes 3 issue cycles instead of 2 (see
// step_uniform) and two warps share a scheduler, which is why the loop reaches
// 0.65 to 0.75 of the FMA rate. n=70, d=64 (width 32), 16 bitstrings: 0.36
// amplitudes/s visiting every tile, 1.34 leaving the zeros out (27 % of the entries
// visited: 0.76 of the HBM copy rate, and 0.59 of the FMA rate by the multiply-adds
// that are executed).
//
// Rescaling: the producer of this pass's input left max(|re|,|im|) of its
// output in maxs[slot]; this pass multiplies its input by 2^s (exact; folded
// into the first step's coefficients) with s chosen so that the maximum lands
// in [0.5, 1), records s in exps[slot+1] and writes its own output maximum to
// maxs[slot+1].
//
// Every mbarrier wait is bounded. A wait that gives up counts once per CTA in
// the device fault word; the warp stops (all its lanes decide together), the
// others then give up too, and the producer waits (bounded) for the tile
// copies it still has in flight before the CTA exits.
#pragma once

#include <cuda.h>

#include "tb_internal.h"

namespace tb {

struct PassParams {
    int h, lo, n;
    int tile_shift;       // log2(tiles visited per batch element) = h - TILE_BITS - skip.n
    int64_t ntiles;       // nbatch << tile_shift
    int runs;             // 1: a CTA works on consecutive tiles, 0: on tiles gridDim.x apart
    int small;            // 1: small tiles (ntiles and tile_shift count them; the host's choice of kernel)
    TileSkip skip;        // which tiles are visited
    WarpSkip warps;       // and which of their warps have something to do
    const StepG* steps;   // the pass's first step
    int xs_step0, xs_q0, xs_step1, xs_q1;
    const uint8_t* bits;  // bitstring of batch element b at bits + b*n
    uint32_t* maxs;       // maxs[b*sstride + slot]
    int32_t* exps;        // exps[b*sstride + slot]
    int64_t sstride;
    int slot;             // slot read; slot+1 written
    int* fault;           // device word: bounded waits that gave up (one per CTA)
    int selftest;         // 1: the producer issues no copies, so every wait gives up
};

__device__ __forceinline__ uint32_t pass_smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Tile bits (13) of a pass and where a consumer thread holds them.
//   LAY_BOT, windows at address bit 0 (tile bits 0..CB-1 = the lowest address
//     bits, window bits 0..M-1; then the chunk): lanes hold tile bits 0..4,
//     registers 5..9, the warp index 10..12;
//   LAY_HIGH, other windows of M <= 9 bits (tile bits 0..3 = the 4 lowest
//     address bits, 4..M+3 the window, then the chunk): registers hold the
//     window's 5 highest bits, lanes its others and tile bit 0; the lanes that
//     are left and the warp index hold tile bits 1..3 and the chunk
//     (thread_base);
//   LAY_LOW3, other windows of 10 bits (tile bits 0..2 = the 3 lowest
//     address bits, rows of 64 bytes): lanes hold tile bits 3..7, registers
//     8..12, the warp index 0..2.
// Every window bit is a lane or register bit in each case.
constexpr int LAY_BOT = 0, LAY_HIGH = 1, LAY_LOW3 = 2;
template <int TYPE_, int M_, bool SMALL_, bool ZW_ = false>
struct Shape {
    static constexpr int TYPE = TYPE_;
    static constexpr int M = M_;
    static constexpr bool SMALL = SMALL_;                 // quarter tiles: 2 consumer warps
    static constexpr bool ZW = ZW_;                       // leaves zero warps out (WarpSkip)
    static constexpr int WARPS = SMALL ? 2 : 8;
    static constexpr int CONSUMERS = 32 * WARPS;
    static constexpr int THREADS = SMALL ? CONSUMERS + 32 : PASS_THREADS;
    static constexpr int STAGES = SMALL ? 1 : 3;          // small tiles: one per CTA
    static constexpr int ENTRIES = 1024 * WARPS;
    static constexpr int ROWL = SMALL ? small_row_log2(TYPE, M) : 0;  // log2 of the parts of a row
    static constexpr bool BOT = bottom_type(TYPE);
    static constexpr int NS = pass_nsteps(TYPE, M);
    static constexpr int XM = pass_xm(TYPE, M);           // step with four variants (-1: none)
    static constexpr int BLK = pass_blk(TYPE, M);         // the turn's 4x4 block (-1: none)
    static constexpr int NB = 2 * NS + (XM >= 0 ? 2 : 0);  // coefficient blocks
    static constexpr int C = BOT ? 0 : high_low_bits(M) - ROWL;  // tile bit of window bit 0
    static constexpr int CB = BOT ? bot_chunk_bits(M) : 0;
    static constexpr int CHL = pass_chunk_log2(TYPE, M) - (SMALL ? SMALL_TILE_LOG2 - ROWL : 0);  // log2 of the chunks of a tile
    static constexpr int LAY = BOT ? LAY_BOT : (M > 9 ? LAY_LOW3 : LAY_HIGH);
    static constexpr int SWZ = BOT || C == 4 ? 128 : (C == 3 ? 64 : 32);  // bytes of a row of the stage
    static constexpr int REG0 = BOT ? 5 : C + M - REG_BITS;  // tile bit of register bit 0
    static constexpr int regpos(int t) { return (t >= REG0 && t < REG0 + REG_BITS) ? t - REG0 : -1; }
    static constexpr int lanepos(int t) {
        if (BOT) return t < 5 ? t : -1;
        if (LAY == LAY_LOW3) return (t >= 3 && t < 8) ? t - 3 : -1;
        return t == 0 ? 0 : (t >= C && t < REG0) ? t - C + 1 : -1;
    }
    static constexpr int tgt(int i) { return C + step_spec(TYPE, M, i).t; }
    static constexpr int ctl(int i) { return step_spec(TYPE, M, i).c < 0 ? -1 : C + step_spec(TYPE, M, i).c; }
    static constexpr bool valid() {
        if (M < MIN_WINDOW || M > (BOT ? MAX_WINDOW : MAX_WINDOW_HIGH)) return false;
        if (SMALL && !has_small_tiles(TYPE, M)) return false;
        for (int j = 0; j < NS; ++j) {
            if (j == BLK) {  // bottom: lanes 0, 1 with control lane 2; top: registers 3, 4 with control register 2
                if (BOT ? (lanepos(tgt(j)) != 0 || lanepos(tgt(j) + 1) != 1 || lanepos(ctl(j)) != 2)
                        : (regpos(tgt(j)) != 3 || regpos(tgt(j) + 1) != 4 || regpos(ctl(j)) != 2))
                    return false;
                continue;
            }
            if (regpos(tgt(j)) < 0 && lanepos(tgt(j)) < 0) return false;
            if (ctl(j) >= 0 && regpos(ctl(j)) < 0 && lanepos(ctl(j)) < 0) return false;
        }
        return true;
    }
};

// Tile coordinate of a consumer thread's register entry 0. LAY_HIGH: tile bits
// of the lanes, then of the warp index; the first four lanes (a half warp's
// accesses) map to four different bank bits, see slot_of.
template <class SH>
__device__ __forceinline__ uint32_t thread_base(uint32_t tid) {
    const uint32_t lane = tid & 31u, warp = tid >> 5;
    if constexpr (SH::LAY == LAY_BOT) return lane | (warp << 10);
    if constexpr (SH::LAY == LAY_LOW3) return (lane << 3) | warp;
    constexpr int BITS[5][8] = {{0, 1, 2, 3, 9, 10, 11, 12},   // M = 5
                                {0, 4, 2, 3, 1, 10, 11, 12},   // 6
                                {0, 4, 5, 3, 1, 2, 11, 12},    // 7
                                {0, 4, 5, 6, 1, 2, 3, 12},     // 8
                                {0, 4, 5, 6, 7, 1, 2, 3}};     // 9
    constexpr int SBITS[5][6] = {{0, 1, 2, 3, 9, 10},  // small tiles; M = 8 and 9 hold 3 and 2 low address bits
                                 {0, 4, 2, 3, 1, 10},
                                 {0, 4, 5, 3, 1, 2},
                                 {0, 3, 4, 5, 1, 2},
                                 {0, 2, 3, 4, 5, 1}};
    uint32_t b = 0;
#pragma unroll
    for (int i = 0; i < (SH::SMALL ? 6 : 8); ++i)
        b |= (tid >> i & 1u) << (SH::SMALL ? SBITS[SH::M < 9 ? SH::M - 5 : 4][i < 6 ? i : 0] : BITS[SH::M < 9 ? SH::M - 5 : 4][i]);
    return b;
}

// ---------------------------------------------------------------------------
// Shared-memory layout of a stage (8-byte slots). The tensor copy writes the
// box in the order of its dimensions, so the stage position of a tile
// coordinate is a permutation of its bits, and the 128-byte swizzle then XORs
// slot bits 1..3 with slot bits 4..6 (16-byte chunk index with the 128-byte
// row index, stage 1024-byte aligned). A half warp's 8-byte accesses are free
// of bank conflicts when its 16 slots differ in bits 0..3 after the swizzle.
//   * windows above bit 0: identity order, so the swizzled bits 0..3 are
//     t0, t1^t4, t2^t5, t3^t6; lanes 0..3 hold tile bit 0 and one of each of
//     the other three pairs, the registers and the warp index the rest: a
//     bijection of the lane bits.
//   * windows at bit 0, per chunk of 2^CB entries: tile bits 0..3, then
//     5..CB-1, then 4; then the chunk (tile bits CB..12). Lanes 0..3 hold
//     tile bits 0..3 and registers bits 5..7, so the swizzled bits are
//     t0, t1^t5, t2^t6, t3^t7: again a bijection of the lane bits.
//   * small tiles of 8- and 9-bit windows: identity order in rows of 64 and 32
//     bytes with their swizzles; lanes 0..3 again reach four different bank
//     bits (M = 8: t0, t3, t4 -> 1, t5 -> 2; M = 9: t0, t2, t3, t4 -> 1).
//   * 10-bit windows above bit 0 (LAY_LOW3): identity order in rows of 64
//     bytes with the 64-byte swizzle (slot bits 1..2 ^= 4..5). Slot bit 0 is
//     the warp's tile bit 0, so a half warp's 16 slots cover 8 bank pairs:
//     two-way conflicts on these passes' stage reads and writes.
// The map is linear over GF(2): for disjoint bit sets slot_of(a | b) =
// slot_of(a) ^ slot_of(b), so a thread's 32 slots are its base slot XOR
// compile-time constants.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr uint32_t swz128(uint32_t s) { return s ^ (((s >> 4) & 7u) << 1); }

// Rows of 64 bytes: slot bits 1..2 ^= 4..5; of 32 bytes: slot bit 1 ^= 4.
__host__ __device__ constexpr uint32_t swz64(uint32_t s) { return s ^ (((s >> 4) & 3u) << 1); }
__host__ __device__ constexpr uint32_t swz32(uint32_t s) { return s ^ (((s >> 4) & 1u) << 1); }

template <class SH>
__host__ __device__ constexpr uint32_t slot_of(uint32_t idx) {
    if (SH::SWZ == 64) return swz64(idx);
    if (SH::SWZ == 32) return swz32(idx);
    constexpr uint32_t MID = SH::BOT ? (1u << (SH::CB - 5)) - 1u : 0u;  // bits 5..CB-1
    return swz128(SH::BOT ? ((idx & 15u) | (((idx >> 5) & MID) << 4) | (((idx >> 4) & 1u) << (SH::CB - 1)) |
                             ((idx >> SH::CB) << SH::CB))
                          : idx);
}

template <class SH, uint32_t J>
struct SlotC {
    static constexpr uint32_t v = slot_of<SH>(J);
};

// ---------------------------------------------------------------------------
// Packed complex arithmetic. A thread's 32 entries are j = k + 16 v (k:
// register bits 0..3, v: register bit 4). They are held "planar" in packed
// pairs P[k] = (re_k, re_(k+16)), Q[k] = (im_k, im_(k+16)), so that one
// __ffma2_rn (sm_100+ paired FP32 FMA) advances two entries that share their
// coefficient. A register step on bit K < 4 with coefficients shared by both
// halves needs 8 paired FMAs per pair of packed registers; a step whose
// control is register bit 4 uses lane-split coefficients; a step whose target
// is register bit 4 mixes the two halves of one packed register. A step on a
// lane bit takes the partner lane's packed registers by shuffles and applies
// the row of G that belongs to this lane's own value of the target bit.
//
// Coefficients are staged in shared memory already packed, 48 float2 per
// (step, bitstring variant):
//   register target, control none / not register bit 4 (KIND_F): for c in
//     0,1: [g00r g00i -g00i g01r g01i -g01i g10r g10i -g10i g11r g11i -g11i],
//     each broadcast to both halves
//   KIND_VC (control = register bit 4): the same 12 values with half c = control
//   KIND_VT (target = register bit 4): for c in 0,1: [Ar Ai -Ai Br Bi -Bi],
//     A = (g00, g11) (own half), B = (g01, g10) (other half)
//   KIND_L (target on a lane): for a (this lane's target value) in 0,1, at
//     24 a: for c in 0,1: [sr si -si or oi -oi] broadcast, s = G[c][a][a],
//     o = G[c][a][1-a]; then at 24 a + 12 the same 6 values with half c =
//     control (control = register bit 4)
// ---------------------------------------------------------------------------
constexpr int VBIT = 4;
constexpr int KIND_F = 0, KIND_VC = 1, KIND_VT = 2, KIND_L = 3, KIND_BL = 4, KIND_BV = 5;
constexpr int CO = 48;  // packed coefficients per (step, variant)

__host__ __device__ __forceinline__ float2 f2x(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }

// out = g0 * a + g1 * b (complex) on planar pairs; cf = 6 packed coefficients
// [g0r g0i -g0i g1r g1i -g1i].
__device__ __forceinline__ void cmac_planar(const float2* cf, float2 aP, float2 aQ, float2 bP, float2 bQ,
                                            float2& oP, float2& oQ) {
    oP = fma2(cf[0], aP, fma2(cf[2], aQ, fma2(cf[3], bP, mul2(cf[5], bQ))));
    oQ = fma2(cf[0], aQ, fma2(cf[1], aP, fma2(cf[3], bQ, mul2(cf[4], bP))));
}

template <int N>
__device__ __forceinline__ void load_cf(float2 (&c)[N], const float2* src, float s) {
    const float4* s4 = reinterpret_cast<const float4*>(src);
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const float4 q = s4[i];
        c[2 * i] = make_float2(q.x * s, q.y * s);
        c[2 * i + 1] = make_float2(q.z * s, q.w * s);
    }
}

// Register target bit K < 4 (pairs of packed registers). CK: -1 none (block
// 0), 0..3 control register bit (block per pair), 4 control = register bit 4
// (lane-split block), 5 control on a lane (block chosen by the caller). The
// pairs of one control value together: half the coefficients live at a time
// (9-bit top turn 11980 cycles per tile in the registers' order, 10360 so).
template <int K, int CK>
__device__ __forceinline__ void step_pairs(float2 (&P)[16], float2 (&Q)[16], const float2* c0, const float2* c1) {
    constexpr bool split = CK >= 0 && CK < 4;
#pragma unroll
    for (int hv = 0; hv < (split ? 2 : 1); ++hv) {
        const float2* c = hv ? c1 : c0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (k & (1 << K)) continue;
            if (split && ((k >> (CK & 3)) & 1) != hv) continue;
            const int k1 = k | (1 << K);
            float2 p0, q0, p1, q1;
            cmac_planar(c, P[k], Q[k], P[k1], Q[k1], p0, q0);
            cmac_planar(c + 6, P[k], Q[k], P[k1], Q[k1], p1, q1);
            P[k] = p0; Q[k] = q0; P[k1] = p1; Q[k1] = q1;
        }
    }
}

// Register target bit 4: the pair is the two halves of one packed register.
template <int CK>
__device__ __forceinline__ void step_halves(float2 (&P)[16], float2 (&Q)[16], const float2* c0, const float2* c1) {
    constexpr bool split = CK >= 0 && CK < 4;
#pragma unroll
    for (int hv = 0; hv < (split ? 2 : 1); ++hv) {
        const float2* c = hv ? c1 : c0;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (split && ((k >> (CK & 3)) & 1) != hv) continue;
            const float2 p = P[k], q = Q[k];
            cmac_planar(c, p, q, swap2(p), swap2(q), P[k], Q[k]);
        }
    }
}

// Lane target (partner lane = lane ^ LM): out = s * own + o * partner. CK as
// for step_pairs; c0 / c1 hold [sr si -si or oi -oi] for control 0 / 1.
template <int CK>
__device__ __forceinline__ void step_lane(float2 (&P)[16], float2 (&Q)[16], const float2 (&c0)[6],
                                          const float2 (&c1)[6], int LM) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const bool hi = (CK >= 0 && CK < 4) ? (((k >> CK) & 1) != 0) : false;
        float2 pp, qp;
        pp.x = __shfl_xor_sync(0xffffffffu, P[k].x, LM);
        pp.y = __shfl_xor_sync(0xffffffffu, P[k].y, LM);
        qp.x = __shfl_xor_sync(0xffffffffu, Q[k].x, LM);
        qp.y = __shfl_xor_sync(0xffffffffu, Q[k].y, LM);
        float2 op, oq;
        if (hi) cmac_planar(c1, P[k], Q[k], pp, qp, op, oq);
        else    cmac_planar(c0, P[k], Q[k], pp, qp, op, oq);
        P[k] = op; Q[k] = oq;
    }
}

// out = sum of four complex products on planar pairs; cf = 12 packed
// coefficients, [re im -im] per input.
__device__ __forceinline__ void cmac4_planar(const float2* cf, float2 aP, float2 aQ, float2 bP, float2 bQ,
                                             float2 cP, float2 cQ, float2 dP, float2 dQ, float2& oP,
                                             float2& oQ) {
    oP = fma2(cf[0], aP, fma2(cf[2], aQ, fma2(cf[3], bP, fma2(cf[5], bQ,
         fma2(cf[6], cP, fma2(cf[8], cQ, fma2(cf[9], dP, mul2(cf[11], dQ))))))));
    oQ = fma2(cf[0], aQ, fma2(cf[1], aP, fma2(cf[3], bQ, fma2(cf[4], bP,
         fma2(cf[6], cQ, fma2(cf[7], cP, fma2(cf[9], dQ, mul2(cf[10], dP))))))));
}

// Turn block on lanes 0, 1 (this lane's block index r = lane & 3): out =
// sum_d B[r][r ^ d] in(lane ^ d); c = [re im -im] of B[r][r ^ d], d = 0..3.
__device__ __forceinline__ void step_block_lanes(float2 (&P)[16], float2 (&Q)[16], const float2 (&c)[12]) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        float2 pp[4], qp[4];
        pp[0] = P[k]; qp[0] = Q[k];
#pragma unroll
        for (int d = 1; d < 4; ++d) {
            pp[d].x = __shfl_xor_sync(0xffffffffu, P[k].x, d);
            pp[d].y = __shfl_xor_sync(0xffffffffu, P[k].y, d);
            qp[d].x = __shfl_xor_sync(0xffffffffu, Q[k].x, d);
            qp[d].y = __shfl_xor_sync(0xffffffffu, Q[k].y, d);
        }
        cmac4_planar(c, pp[0], qp[0], pp[1], qp[1], pp[2], qp[2], pp[3], qp[3], P[k], Q[k]);
    }
}

// Turn block on registers 3 and 4 (register 4 = the packed pair's halves),
// control register 2: packed registers k and k | 8 (k < 8) form the block's
// four entries; cf = the variant's 48 coefficients (24 per control value).
__device__ __forceinline__ void step_block_regs(float2 (&P)[16], float2 (&Q)[16], const float2* cf) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        float2 cc[24];
        load_cf(cc, cf + 24 * c, 1.0f);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
            const int k0 = kk | (c << 2), k1 = k0 | 8;
            const float2 aP = P[k0], aQ = Q[k0], bP = P[k1], bQ = Q[k1];
            const float2 sP = swap2(aP), sQ = swap2(aQ), tP = swap2(bP), tQ = swap2(bQ);
            cmac4_planar(cc, aP, aQ, sP, sQ, bP, bQ, tP, tQ, P[k0], Q[k0]);
            cmac4_planar(cc + 12, aP, aQ, sP, sQ, bP, bQ, tP, tQ, P[k1], Q[k1]);
        }
    }
}

template <class SH>
__host__ __device__ constexpr int step_kind(int i) {
    if (i == SH::BLK) return SH::BOT ? KIND_BL : KIND_BV;
    const int K = SH::regpos(SH::tgt(i));
    if (K < 0) return KIND_L;
    if (K == VBIT) return KIND_VT;
    if (SH::ctl(i) >= 0 && SH::regpos(SH::ctl(i)) == VBIT) return KIND_VC;
    return KIND_F;
}

// Steps whose coefficients come from the kernel's parameters instead of shared
// memory: steps on a register bit that no lane bit controls and no output bit
// changes, so that they are the same for every thread and bitstring. A paired
// FMA takes 3.0 issue cycles with three fresh register pairs and 2.1 with the
// coefficient in the constant bank (a coefficient that several FMAs in a row
// share: 2.2, but no order of the steps' FMAs made ptxas keep it). Consumer loop
// alone, cycles per tile: 9-bit forward window 6030 -> 5620, reversed 6510 -> 6100,
// 7-bit top turn 7900 -> 7320, 9-bit top turn 11150 -> 10360, 8-bit window forward
// 5300 -> 4860, 10-bit bottom turn 13150 -> 13120 (its lane steps and block
// dominate). n=28, d=42, dense gates, 16 bitstrings: 6.00 -> 5.78 ms; n=70, d=56,
// two bitstrings: 131.8 -> 128.2 ms.
// Not the first step, which carries the rescale; small tiles have one tile per
// CTA, where the time is set-up and latency (367 and 361 us on n=33, d=35, no
// difference between runs), and smaller parameters launch faster.
template <class SH>
__host__ __device__ constexpr bool step_uniform(int i) {
    if (SH::SMALL || i == 0 || i == SH::BLK || output_step(SH::TYPE, SH::M, i)) return false;
    return SH::regpos(SH::tgt(i)) >= 0 && (SH::ctl(i) < 0 || SH::regpos(SH::ctl(i)) >= 0);
}
template <class SH>
__host__ __device__ constexpr int uniform_index(int n) {  // uniform steps before step n
    int u = 0;
    for (int i = 0; i < n; ++i) u += step_uniform<SH>(i) ? 1 : 0;
    return u;
}
constexpr int UCO = 24;  // their packed coefficients
template <class SH>
struct PassConst {
    float2 c[uniform_index<SH>(SH::NS) > 0 ? uniform_index<SH>(SH::NS) : 1][UCO];
};

template <class SH>
__host__ __device__ constexpr uint64_t step_kinds() {
    uint64_t k = 0;
    static_assert(3 * SH::NS <= 64, "three kind bits per step");
    for (int i = 0; i < SH::NS; ++i) k |= (uint64_t)step_kind<SH>(i) << (3 * i);
    return k;
}

template <class SH>
__host__ __device__ constexpr uint32_t uniform_mask() {
    uint32_t m = 0;
    for (int i = 0; i < SH::NS; ++i) m |= (step_uniform<SH>(i) ? 1u : 0u) << i;
    return m;
}

// The packed coefficients of a step on a register bit (KIND_F, _VC, _VT) from
// its blocks g[c*4 + a'*2 + s].
__host__ __device__ inline void pack_register_step(int kind, const float2* g, float2* o) {
    if (kind == KIND_F) {
        for (int c = 0; c < 2; ++c)
            for (int e = 0; e < 4; ++e) {
                const float2 z = g[c * 4 + e];
                o[c * 12 + 3 * e + 0] = f2x(z.x);
                o[c * 12 + 3 * e + 1] = f2x(z.y);
                o[c * 12 + 3 * e + 2] = f2x(-z.y);
            }
    } else if (kind == KIND_VC) {
        for (int e = 0; e < 4; ++e) {
            const float2 z0 = g[e], z1 = g[4 + e];
            o[3 * e + 0] = make_float2(z0.x, z1.x);
            o[3 * e + 1] = make_float2(z0.y, z1.y);
            o[3 * e + 2] = make_float2(-z0.y, -z1.y);
        }
    } else if (kind == KIND_VT) {
        for (int c = 0; c < 2; ++c) {
            const float2 A0 = g[c * 4 + 0], A1 = g[c * 4 + 3];  // own half: g00 (lo), g11 (hi)
            const float2 B0 = g[c * 4 + 1], B1 = g[c * 4 + 2];  // other half: g01 (lo), g10 (hi)
            o[c * 12 + 0] = make_float2(A0.x, A1.x);
            o[c * 12 + 1] = make_float2(A0.y, A1.y);
            o[c * 12 + 2] = make_float2(-A0.y, -A1.y);
            o[c * 12 + 3] = make_float2(B0.x, B1.x);
            o[c * 12 + 4] = make_float2(B0.y, B1.y);
            o[c * 12 + 5] = make_float2(-B0.y, -B1.y);
        }
    }
}

// Stage the packed coefficients of every step and variant into shared memory.
// Blocks 2 i + x: step i, variant x; blocks 2 NS + x: the four-variant
// step's (the top block's) variants 2 + x. Turn blocks (raw float2[variant][c][q'][q] over
// BLK_ENTRIES table entries):
//   KIND_BL (lanes 0, 1; control lane 2; no output-bit dependence): blocks
//     2 i and 2 i + 1 hold, at 12 (4 c + r), [re im -im] of B[c][r][r ^ d]
//     for d = 0..3, broadcast (r = the lane's block index)
//   KIND_BV (registers 3, 4; control register 2): per variant, at 24 c + 12 b
//     (output register: block bit t = b), four packed pairs for the inputs
//     [register t=0, swapped, register t=1, swapped]: (B[b][a], B[b+2][a+2])
//     and (B[b][a+2], B[b+2][a]) for a = 0, 1, each as [re im -im]
template <class SH>
__device__ __forceinline__ void stage_coefficients(const StepG* steps, float2* sc, uint32_t tid) {
    constexpr uint64_t KINDS = step_kinds<SH>();
    constexpr uint32_t UNIFORM = uniform_mask<SH>();
    for (int w = tid; w < SH::NB; w += SH::THREADS) {
        const int i = w < 2 * SH::NS ? w >> 1 : SH::XM, x = w & 1;
        if ((UNIFORM >> i) & 1u) continue;
        float2* o = sc + w * CO;
        for (int e = 0; e < CO; ++e) o[e] = make_float2(0.f, 0.f);
        const int kind = (int)((KINDS >> (3 * i)) & 7u);
        if (kind == KIND_BL || kind == KIND_BV) {
            const float2* raw = &steps[pass_entry(SH::TYPE, SH::M, i)].g[0][0];
            auto Bq = [&](int v, int c, int r, int q) { return raw[((v * 2 + c) * 4 + r) * 4 + q]; };
            if (kind == KIND_BL) {  // block w - 2 i = control value c
                for (int r = 0; r < 4; ++r)
                    for (int d = 0; d < 4; ++d) {
                        const float2 z = Bq(0, x, r, r ^ d);
                        o[12 * r + 3 * d + 0] = f2x(z.x);
                        o[12 * r + 3 * d + 1] = f2x(z.y);
                        o[12 * r + 3 * d + 2] = f2x(-z.y);
                    }
            } else {
                const int v = x + (w < 2 * SH::NS ? 0 : 2);
                for (int c = 0; c < 2; ++c)
                    for (int b = 0; b < 2; ++b)
                        for (int a = 0; a < 2; ++a)
                            for (int sw = 0; sw < 2; ++sw) {
                                const float2 lo = Bq(v, c, b, sw ? a + 2 : a), hi = Bq(v, c, b + 2, sw ? a : a + 2);
                                float2* t = o + 24 * c + 12 * b + 6 * a + 3 * sw;
                                t[0] = make_float2(lo.x, hi.x);
                                t[1] = make_float2(lo.y, hi.y);
                                t[2] = make_float2(-lo.y, -hi.y);
                            }
            }
            continue;
        }
        const float2* g = steps[pass_entry(SH::TYPE, SH::M, i)].g[x];  // [c*4 + a'*2 + s]
        if (kind != KIND_L) {
            pack_register_step(kind, g, o);
        } else {
            for (int a = 0; a < 2; ++a) {
                float2* oa = o + 24 * a;
                for (int c = 0; c < 2; ++c) {
                    const float2 sv = g[c * 4 + a * 2 + a], ov = g[c * 4 + a * 2 + (1 - a)];
                    const float v[6] = {sv.x, sv.y, -sv.y, ov.x, ov.y, -ov.y};
                    for (int e = 0; e < 6; ++e) {
                        oa[c * 6 + e] = f2x(v[e]);
                        if (c == 0) oa[12 + e].x = v[e];
                        else        oa[12 + e].y = v[e];
                    }
                }
            }
        }
    }
}

// Registers <-> shared stage: entry j of a thread sits at tile coordinate
// thread_base | j << REG0, i.e. slot base ^ SlotC<j << REG0>.
template <class SH, int J>
__device__ __forceinline__ void smem_read_j(float2 (&P)[16], float2 (&Q)[16], const float2* tile, uint32_t sb) {
    if constexpr (J < 32) {
        const float2 e = tile[sb ^ SlotC<SH, ((uint32_t)J << SH::REG0)>::v];
        if constexpr (J < 16) { P[J].x = e.x; Q[J].x = e.y; }
        else                  { P[J - 16].y = e.x; Q[J - 16].y = e.y; }
        smem_read_j<SH, J + 1>(P, Q, tile, sb);
    }
}

template <class SH, int J>
__device__ __forceinline__ void smem_write_j(const float2 (&P)[16], const float2 (&Q)[16], float2* tile,
                                             uint32_t sb) {
    if constexpr (J < 32) {
        tile[sb ^ SlotC<SH, ((uint32_t)J << SH::REG0)>::v] =
            J < 16 ? make_float2(P[J & 15].x, Q[J & 15].x) : make_float2(P[J & 15].y, Q[J & 15].y);
        smem_write_j<SH, J + 1>(P, Q, tile, sb);
    }
}

template <class SH, int I>
__device__ __forceinline__ void apply_step(float2 (&P)[16], float2 (&Q)[16], const float2* sc,
                                           const PassConst<SH>& pc, uint32_t xmask, float scale, uint32_t tid) {
    constexpr int T = SH::tgt(I), CB = SH::ctl(I);
    constexpr int kind = step_kind<SH>(I);
    // control: -1 none, 0..4 register bit, 5 on a lane (the same for all of
    // this thread's entries)
    constexpr int CK = CB < 0 ? -1 : (SH::regpos(CB) >= 0 ? SH::regpos(CB) : 5);
    const uint32_t lane = tid & 31u;
    const float s = (I == 0) ? scale : 1.0f;
    asm volatile("" ::: "memory");  // load each step's coefficients just before it
    const float2* cf;
    if constexpr (I == SH::XM) {  // variant x_a + 2 x_b
        cf = sc + (((xmask >> XM_HIGH_BIT) & 1u) ? 2 * SH::NS : I * 2) * CO + (int)((xmask >> I) & 1u) * CO;
    } else {
        cf = sc + (I * 2 + (int)((xmask >> I) & 1u)) * CO;
    }
    if constexpr (kind == KIND_BL) {
        float2 c[12];
        static_assert(I > 0, "the first step carries the rescale");
        load_cf(c, sc + (I * 2 + (int)((lane >> 2) & 1u)) * CO + (lane & 3u) * 12u, 1.0f);  // control lane 2
        step_block_lanes(P, Q, c);
    } else if constexpr (kind == KIND_BV) {
        static_assert(I > 0 && I == SH::XM, "the top block has four variants and no rescale");
        step_block_regs(P, Q, cf);
    } else if constexpr (kind == KIND_L) {
        constexpr int L = SH::lanepos(T);
        static_assert(L >= 0, "lane target");
        const float2* ca = cf + 24 * ((lane >> L) & 1u);
        float2 c0[6], c1[6];
        if constexpr (CK == 5) {
            load_cf(c0, ca + 6 * ((lane >> SH::lanepos(CB)) & 1u), s);
        } else if constexpr (CK == 4) {
            load_cf(c0, ca + 12, s);
        } else {
            load_cf(c0, ca, s);
            if constexpr (CK >= 0) load_cf(c1, ca + 6, s);
        }
        step_lane<(CK == 4 || CK == 5) ? -1 : CK>(P, Q, c0, c1, 1 << L);
    } else if constexpr (step_uniform<SH>(I)) {
        const float2* c = pc.c[uniform_index<SH>(I)];
        if constexpr (kind == KIND_VT) step_halves<CK>(P, Q, c, c + 12);
        else step_pairs<SH::regpos(T), CK>(P, Q, c, c + 12);
    } else {
        constexpr int K = SH::regpos(T);
        float2 c0[12], c1[12];
        if constexpr (CK == 5) {
            load_cf(c0, cf + 12 * ((lane >> SH::lanepos(CB)) & 1u), s);
        } else {
            load_cf(c0, cf, s);
        }
        if constexpr (CK >= 0 && CK < 4) load_cf(c1, cf + 12, s);
        if constexpr (kind == KIND_VT) {
            step_halves<(CK == 5) ? -1 : CK>(P, Q, c0, c1);
        } else {
            step_pairs<K, (CK == 5) ? -1 : CK>(P, Q, c0, c1);
        }
    }
}

template <class SH, int I>
__device__ __forceinline__ void run_steps(float2 (&P)[16], float2 (&Q)[16], const float2* sc,
                                          const PassConst<SH>& pc, uint32_t xmask, float scale, uint32_t tid) {
    if constexpr (I < SH::NS) {
        apply_step<SH, I>(P, Q, sc, pc, xmask, scale, tid);
        run_steps<SH, I + 1>(P, Q, sc, pc, xmask, scale, tid);
    }
}

__device__ __forceinline__ void flush_max(float m, uint32_t* dst) {
    // m >= 0: floats compare like their bits
    const uint32_t u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) atomicMax(dst, u);
}

// Power of two that brings a maximum m into [0.5, 1); 0 for m == 0.
__device__ __forceinline__ int rescale_exp(float m) {
    if (!(m > 0.0f) || !isfinite(m)) return 0;
    int e;
    frexpf(m, &e);
    return max(-100, min(100, -e));
}

// ---------------------------------------------------------------------------
// mbarriers and tensor copies (PTX)
// ---------------------------------------------------------------------------
constexpr uint32_t PASS_WAIT_TRIES = 1u << 24;    // far beyond any tile's copy or compute time
constexpr uint32_t PASS_SELFTEST_TRIES = 1u << 10;

__device__ __forceinline__ void pbar_init(uint32_t a, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(a), "r"(count) : "memory");
}

__device__ __forceinline__ void pbar_arrive(uint32_t a) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(a) : "memory");
}

__device__ __forceinline__ void pbar_expect_tx(uint32_t a, uint32_t bytes) {
    asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n" ::"r"(a),
                 "r"(bytes)
                 : "memory");
}

// Bounded wait for the phase with the given parity; false if it gave up.
__device__ __forceinline__ bool pbar_wait(uint32_t a, uint32_t parity, uint32_t tries) {
    for (uint32_t it = 0; it < tries; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_load_tile(uint32_t dst, const CUtensorMap* m, int c3, int c4, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %2, %2, %3, %4}], [%5];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(m)), "r"(0), "r"(c3), "r"(c4), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_store_tile(const CUtensorMap* m, int c3, int c4, uint32_t src) {
    asm volatile(
        "cp.async.bulk.tensor.5d.global.shared::cta.tile.bulk_group [%0, {%1, %1, %1, %2, %3}], [%4];\n" ::"l"(
            reinterpret_cast<uint64_t>(m)),
        "r"(0), "r"(c3), "r"(c4), "r"(src)
        : "memory");
    asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}

__device__ __forceinline__ void tma_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory"); }
__device__ __forceinline__ void tma_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// Tensor-map coordinates (dimensions 3 and 4) of the chunk that this lane moves
// of visited tile gt (the whole producer warp; col = this lane's column of the
// tile map, chunk = the XOR of the columns of the lane's own bits). Windows at
// bit 0: dimension 3 = the chunk index with the batch element. Other windows:
// dimension 3 = the address bits between the low bits and the window,
// dimension 4 = the bits above the window and the batch element.
template <class SH>
__device__ __forceinline__ void tile_coords(const PassParams& p, int64_t gt, uint32_t col, uint32_t lane,
                                            uint32_t chunk, int& c3, int& c4) {
    const int64_t b = gt >> p.tile_shift;
    const uint32_t u = (uint32_t)(gt & (((int64_t)1 << p.tile_shift) - 1));
    int64_t t = tile_of_warp(p.skip.base, col, lane, (u >> SH::ROWL) << SH::CHL) ^ chunk;
    if constexpr (SH::ROWL > 0) t = (t << SH::ROWL) | (u & ((1u << SH::ROWL) - 1u));  // part of the rows
    if constexpr (SH::BOT) {
        c3 = (int)((b << (p.h - SH::CB)) + t);
        c4 = 0;
    } else {
        const int nl = p.lo - SH::C;
        c3 = (int)(t & (((int64_t)1 << nl) - 1));
        c4 = (int)((b << (p.h - p.lo - SH::M)) + (t >> nl));
    }
}

// Tile-map columns of the chunk that warp w works on (8-bit windows: two chunks
// per tile, the warp index's highest bit; 9-bit windows: one).
template <class SH>
__device__ __forceinline__ uint32_t chunk_of_warp(uint32_t col, uint32_t w) {
    if constexpr (SH::CHL == 0) return 0u;
    const uint32_t c0 = __shfl_sync(0xffffffffu, col, 0);
    return w >> 2 & 1u ? c0 : 0u;
}

template <class SH>
constexpr int pass_smem_bytes() {
    return 1024 + SH::STAGES * SH::ENTRIES * 8 + SH::NB * CO * 8 + 2 * SH::STAGES * 8 + 16;
}

template <class SH>
__global__ void __launch_bounds__(SH::THREADS, SH::SMALL ? SMALL_CTAS_PER_SM : PASS_CTAS_PER_SM)
    pass_kernel(const __grid_constant__ PassParams p, const __grid_constant__ CUtensorMap tmap,
                const __grid_constant__ PassConst<SH> pc) {
    static_assert(SH::valid(), "invalid pass shape");
    static_assert(SH::NS <= XM_HIGH_BIT, "variant mask: one bit per step, bit XM_HIGH_BIT for the four-variant step");
    constexpr int STAGES = SH::STAGES;
    constexpr uint32_t TILE_BYTES = SH::ENTRIES * 8u;
    extern __shared__ __align__(16) uint8_t dsm[];
    uint8_t* base = dsm + ((1024u - (pass_smem_u32(dsm) & 1023u)) & 1023u);
    float2* stages = reinterpret_cast<float2*>(base);
    float2* sc = stages + STAGES * SH::ENTRIES;
    uint64_t* bars = reinterpret_cast<uint64_t*>(sc + SH::NB * CO);  // full[3], done[3]
    int* s_abort = reinterpret_cast<int*>(bars + 2 * STAGES);
    const uint32_t tid = threadIdx.x;
    const uint32_t full0 = pass_smem_u32(bars), done0 = full0 + 8 * STAGES;
    const uint32_t stage0 = pass_smem_u32(stages);

    // tiles first, first + step, ... of this CTA (grid <= ntiles)
    const int64_t first = p.runs ? p.ntiles * blockIdx.x / gridDim.x : blockIdx.x;
    const int64_t step = p.runs ? 1 : gridDim.x;
    const int64_t ntl = p.runs ? p.ntiles * (blockIdx.x + 1) / gridDim.x - first
                               : (p.ntiles - 1 - first) / gridDim.x + 1;
    const uint32_t tries = p.selftest ? PASS_SELFTEST_TRIES : PASS_WAIT_TRIES;
    const uint32_t lane = tid & 31u;
    const uint32_t col = tile_col(p.skip, lane);
    // copies of a tile: one per chunk, issued by as many lanes
    constexpr uint32_t PART = TILE_BYTES >> SH::CHL;
    const bool mover = lane < (1u << SH::CHL);
    uint32_t chunk = 0;
#pragma unroll
    for (int i = 0; i < SH::CHL; ++i) {
        const uint32_t ci = __shfl_sync(0xffffffffu, col, i);
        if (lane >> i & 1u) chunk ^= ci;
    }
    int t3[STAGES], t4[STAGES];  // producer: coordinates of the tile in each stage

    // The producer warp (the first of the last warpgroup) works on tile
    // coordinates together; its lane 0 sets the barriers up and issues every
    // copy. The first loads do not wait for the coefficients.
    if ((tid >> 5) == SH::WARPS) {
        if (lane == 0) {
            asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&tmap)) : "memory");
            for (int s = 0; s < STAGES; ++s) {
                pbar_init(full0 + 8 * s, 1);
                pbar_init(done0 + 8 * s, SH::WARPS);
            }
            *s_abort = 0;
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        }
        grid_wait();
        if (!p.selftest)
            for (int k = 0; k < ntl && k < STAGES; ++k) {
                tile_coords<SH>(p, first + k * step, col, lane, chunk, t3[k], t4[k]);
                if (lane == 0) pbar_expect_tx(full0 + 8 * k, TILE_BYTES);
                __syncwarp();
                if (mover) tma_load_tile(stage0 + (uint32_t)k * TILE_BYTES + lane * PART, &tmap, t3[k], t4[k], full0 + 8 * k);
            }
    }
    // One tile per CTA: the next pass's CTAs start on free SMs at once. With more
    // tiles a CTA of the next pass would only hold the SM that another CTA of
    // this pass leaves (or that another stream's work could use), so the release
    // waits for the end. Measured (us, none / at the end / at once): n=33, d=35,
    // one bitstring 459 / 420 / 406; n=61, d=32, 200 bitstrings 4461 / 4393 /
    // 4413; n=28, d=42, 16 bitstrings 6643 / 6680 / 6906; plain launches 525,
    // 4619, 6796.
    const bool one_tile = p.ntiles <= gridDim.x;
    if (one_tile) grid_release();
    stage_coefficients<SH>(p.steps, sc, tid);
    grid_wait();  // every thread: the boundary and the rescaling state are the predecessor's
    __syncthreads();

    static_assert(PASS_THREADS - PASS_CONSUMERS == 128, "one producer warpgroup");
    static_assert((PASS_THREADS - PASS_CONSUMERS) * PASS_PRODUCER_REGS + PASS_CONSUMERS * PASS_CONSUMER_REGS <=
                      PASS_THREADS * (65536 / PASS_THREADS / 8 * 8),
                  "register split exceeds the launch's registers");
    if (tid >= SH::CONSUMERS) {
        // ---------------- producer: one warp (of the last warpgroup)
        if constexpr (!SH::SMALL) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(PASS_PRODUCER_REGS));
        if ((tid >> 5) != SH::WARPS) return;
        int64_t last_load[STAGES];  // tile index k of the latest load per stage (-1: none)
        for (int st = 0; st < STAGES; ++st) last_load[st] = !p.selftest && st < ntl ? st : -1;
        int s = 0;
        uint32_t ph = 0;
        for (int64_t k = 0; k < ntl; ++k) {
            int n3 = 0, n4 = 0;  // the stage's next tile, worked out while the consumers are busy
            if (k + STAGES < ntl) tile_coords<SH>(p, first + (k + STAGES) * step, col, lane, chunk, n3, n4);
            const bool gave_up = !pbar_wait(done0 + 8 * s, ph, tries);
            if (__any_sync(0xffffffffu, gave_up)) {
                if (lane == 0 && atomicExch(s_abort, 1) == 0) atomicAdd(p.fault, 1);
                break;
            }
            if (mover) tma_store_tile(&tmap, t3[s], t4[s], stage0 + (uint32_t)s * TILE_BYTES + lane * PART);
            if (k + STAGES < ntl) {
                if (mover) tma_wait_read_all();  // the stores have read the stage
                if (lane == 0) pbar_expect_tx(full0 + 8 * s, TILE_BYTES);
                __syncwarp();
                if (mover) tma_load_tile(stage0 + (uint32_t)s * TILE_BYTES + lane * PART, &tmap, n3, n4, full0 + 8 * s);
                last_load[s] = k + STAGES;
                t3[s] = n3;
                t4[s] = n4;
            }
            __syncwarp();
            if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
        if (mover) tma_wait_all();
        __syncwarp();
        if (lane == 0 && *(volatile int*)s_abort) {
            // loads still in flight must land before the CTA's shared memory goes
            for (int st = 0; st < STAGES; ++st)
                if (last_load[st] >= 0)
                    (void)pbar_wait(full0 + 8 * st, (uint32_t)((last_load[st] / STAGES) & 1), PASS_WAIT_TRIES);
        }
        return;
    }

    // ---------------- consumers: 8 (small tiles: 2) independent warps
    if constexpr (!SH::SMALL) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(PASS_CONSUMER_REGS));
    float runmax = 0.0f;
    int64_t cur_b = -1;
    int cur_s = 0;
    float scale = 1.0f;
    uint32_t xmask = 0;
    const int64_t tmask = ((int64_t)1 << p.tile_shift) - 1;
    uint32_t sb = slot_of<SH>(thread_base<SH>(tid));
    // Zero warps: a warp whose 1024 entries are zero passes the tile on. Which
    // they are changes with the tile at most through its address, so the warps
    // take turns (warp w works as warp w ^ k on tile k): otherwise the same
    // schedulers would idle in every tile. n=61, d=32, 200 bitstrings 3.54 ->
    // 3.33 ms. A kernel of its own: in the common one it took 2 % of the passes
    // without zero warps.
    uint32_t wout = 0, wmask = 0;
    uint32_t wslot[3] = {0, 0, 0};
    if constexpr (SH::ZW) {
        if (lane < (uint32_t)p.warps.n) {
            wout = p.warps.out[lane];
            wmask = p.warps.warp[lane];
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) wslot[i] = slot_of<SH>(thread_base<SH>(32u << i));
    }
    const uint32_t sb0 = sb;
    // A bitstring's rescaling maximum and output bits, read while the tile before
    // its first one is worked on: reading the state on the spot put two global
    // latencies into every change of bitstring (n=61, d=32, 200 bitstrings: 3.90
    // -> 3.72 ms; n=30, d=40, 32: 5.30 -> 4.81 ms).
    uint32_t next_max = 0;
    uint32_t next_x = 0;
    auto read_state = [&](int64_t b) {
        next_max = p.maxs[b * p.sstride + p.slot];
        const uint8_t* xb = p.bits + b * p.n;
        next_x = 0;
        if (p.xs_step0 >= 0) next_x |= xb[p.xs_q0];
        if (p.xs_step1 >= 0) next_x |= (uint32_t)xb[p.xs_q1] << 8;
    };
    if (ntl > 0) read_state(first >> p.tile_shift);
    int s = 0;
    uint32_t ph = 0;
    for (int64_t k = 0; k < ntl; ++k) {
        const int64_t gt = first + k * step;
        const int64_t b = gt >> p.tile_shift;
        const int64_t t = gt & tmask;
        if (b != cur_b) {
            if (cur_b >= 0) flush_max(runmax, p.maxs + cur_b * p.sstride + p.slot + 1);
            runmax = 0.0f;
            cur_b = b;
            cur_s = rescale_exp(__uint_as_float(next_max));
            scale = ldexpf(1.0f, cur_s);
            xmask = 0;
            if (p.xs_step0 >= 0) xmask |= (next_x & 0xffu ? 1u : 0u) << p.xs_step0;
            if (p.xs_step1 >= 0) xmask |= (next_x >> 8 ? 1u : 0u) << p.xs_step1;
        }
        if (k + 1 < ntl) {
            const int64_t bn = (gt + step) >> p.tile_shift;
            if (bn != b) read_state(bn);
        }
        const bool gave_up = !pbar_wait(full0 + 8 * s, ph, tries);
        if (__any_sync(0xffffffffu, gave_up)) {  // the whole warp stops
            if ((tid & 31u) == 0 && atomicExch(s_abort, 1) == 0) atomicAdd(p.fault, 1);
            break;
        }
        bool idle = false;
        if constexpr (SH::ZW) {
            const uint32_t turn = (uint32_t)k & 7u, w = (tid >> 5) ^ turn;
            sb = sb0 ^ (turn & 1u ? wslot[0] : 0u) ^ (turn & 2u ? wslot[1] : 0u) ^ (turn & 4u ? wslot[2] : 0u);
            const uint32_t ti = tile_of_warp(p.skip.base, col, lane, (uint32_t)t << SH::CHL) ^ chunk_of_warp<SH>(col, w);
            idle = __any_sync(0xffffffffu, ((uint32_t)__popc(ti & wout) + (uint32_t)__popc(w & wmask & 7u) + (wmask >> 3)) & 1u);
        }
        if (t == 0 && tid == 0) p.exps[b * p.sstride + p.slot + 1] = cur_s;

        if (idle) {
            if (lane == 0) pbar_arrive(done0 + 8 * s);
            if (++s == STAGES) { s = 0; ph ^= 1u; }
            continue;
        }
        float2* tile = stages + s * SH::ENTRIES;
        float2 P[16], Q[16];
        smem_read_j<SH, 0>(P, Q, tile, sb);
        run_steps<SH, 0>(P, Q, sc, pc, xmask, scale, tid);
#pragma unroll
        for (int j = 0; j < 16; ++j)
            runmax = fmaxf(runmax, fmaxf(fmaxf(fabsf(P[j].x), fabsf(P[j].y)), fmaxf(fabsf(Q[j].x), fabsf(Q[j].y))));
        smem_write_j<SH, 0>(P, Q, tile, sb);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // visible to the tensor store
        __syncwarp();
        if ((tid & 31u) == 0) pbar_arrive(done0 + 8 * s);
        if (++s == STAGES) { s = 0; ph ^= 1u; }
    }
    if (cur_b >= 0) flush_max(runmax, p.maxs + cur_b * p.sstride + p.slot + 1);
    if (!one_tile) grid_release();
}

// Launchers, one translation unit per pass type (pass_t<type>.cu). host_steps:
// the pass's entries of the pass-step table in host memory (p.steps is its copy
// on the device).
cudaError_t launch_pass_t0(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);
cudaError_t launch_pass_t1(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);
cudaError_t launch_pass_t2(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);
cudaError_t launch_pass_t3(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);
cudaError_t launch_pass_t4(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);
cudaError_t launch_pass_t5(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);
cudaError_t launch_pass_t6(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                           cudaStream_t st);

template <class SH>
cudaError_t launch_shape(const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,
                         cudaStream_t st) {
    if constexpr (!SH::valid()) {
        return cudaErrorInvalidValue;
    } else {
        constexpr int smem = pass_smem_bytes<SH>();
        static_assert(smem <= 227 * 1024, "pass kernel shared memory");
        cudaError_t e = cudaFuncSetAttribute(pass_kernel<SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        PassConst<SH> pc{};
        for (int i = 0; i < SH::NS; ++i) {
            if (!step_uniform<SH>(i)) continue;
            if (p.xs_step0 == i || p.xs_step1 == i) return cudaErrorInvalidValue;  // output_step excludes it
            pack_register_step(step_kind<SH>(i), host_steps[pass_entry(SH::TYPE, SH::M, i)].g[0],
                               pc.c[uniform_index<SH>(i)]);
        }
        return launch_after(pass_kernel<SH>, grid, SH::THREADS, smem, st, p, m, pc);
    }
}

template <int TYPE, int M>
cudaError_t launch_one(const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid, cudaStream_t st) {
    if (p.small) return launch_shape<Shape<TYPE, M, true>>(p, host_steps, m, grid, st);
    if constexpr (warp_addr_bits(TYPE, M) > 0) {
        if (p.warps.n > 0) return launch_shape<Shape<TYPE, M, false, true>>(p, host_steps, m, grid, st);
    }
    return launch_shape<Shape<TYPE, M, false>>(p, host_steps, m, grid, st);
}

#define TB_DEFINE_LAUNCH_PASS(TYPE, NAME)                                                      \
    cudaError_t NAME(int M, const PassParams& p, const StepG* host_steps, const CUtensorMap& m, int grid,  \
                     cudaStream_t st) {                                                   \
        switch (M) {                                                                          \
            case 5: return launch_one<TYPE, 5>(p, host_steps, m, grid, st);               \
            case 6: return launch_one<TYPE, 6>(p, host_steps, m, grid, st);               \
            case 7: return launch_one<TYPE, 7>(p, host_steps, m, grid, st);               \
            case 8: return launch_one<TYPE, 8>(p, host_steps, m, grid, st);               \
            case 9: return launch_one<TYPE, 9>(p, host_steps, m, grid, st);               \
            case 10: return launch_one<TYPE, 10>(p, host_steps, m, grid, st);             \
            default: return cudaErrorInvalidValue;                                            \
        }                                                                                     \
    }

}  // namespace tb
