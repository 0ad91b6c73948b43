// Host-side lengths of the rings in shared memory that the tensor-core kernels' roles hand blocks round in (plain C++, no CUDA).
#pragma once

namespace bpdq {

constexpr int kTsGroups = 4;                          // decode groups of the kernel for up to 128 tokens; they take blocks in turn
constexpr int kTsIssuers = 2;                         // its MMA issuers; blocks alternate between them
constexpr int kTsSmem = 227 * 1024;
constexpr int kTsMaxSX = 8, kTsMaxSP = 24;

constexpr int ts_plane_bytes(int K) { return K * 2048; }
constexpr int ts_coef_bytes(int K) { return (K + 1) * 256; }
constexpr int ts_slot_bytes(int K) { return ts_plane_bytes(K) + 2 * ts_coef_bytes(K); }

struct TsRings {
    int sx, sp;                                       // slots of the x ring and of the packed ring
};

// `cols` token columns (a multiple of 16, at most 128).  The x ring takes as many blocks as 128 KB hold, four to eight, the
// packed ring the rest of shared memory, eight slots or more.
//
// Both lengths are even.  A wait by parity is right only if the barrier's phase before the awaited one is over when the wait
// begins; else it passes at once.  x slots: with an even length a slot belongs to one issuer, which has waited for every use of
// it.  Packed slots: the group that waits for block q has seen its A slot free for block q - 4, so the MMAs of block q - 8 are
// complete, and with them, in the order of its commits, every earlier block of THAT issuer: q - 8, q - 10, ...  With an even
// length of at least eight the slot's last use, block q - sp, is among them, so its copy has landed.  With an odd one it
// belongs to the other issuer, which may be any way behind when that block's copy is late (9 slots at K = 4 with 128 tokens).
constexpr TsRings ts_rings(int K, int cols) {
    int sx = 128 * 1024 / (cols * 256) / 2 * 2;
    if (sx > kTsMaxSX) sx = kTsMaxSX;
    int sp = (kTsSmem - 3072 - sx * cols * 256) / ts_slot_bytes(K) / 2 * 2;   // 3072: alignment slack, barriers
    if (sp > kTsMaxSP) sp = kTsMaxSP;
    return {sx, sp};
}

// Work split of the kernel for up to 128 tokens.  `tiles` row tiles with `units` 128-column blocks in all; rows of one length have
// `nb0` blocks, nb0 = 0 says that the linears differ in length.  CTA b of `grid` takes the units [share(b), share(b + 1)) of the cut
// ones, share(s) = cut_begin + cut_units / cut_step * s / grid * cut_step, and the whole tiles b, b + grid, ... below cut_begin.
struct TsSplit {
    int grid, whole, cut_begin, cut_units, cut_step;
};
constexpr int kTsMinCut = 16;                         // blocks per row from which tiles are shared between CTAs
constexpr int kTsMinShare = 8;                        // blocks of a share at least (a share of a tile costs a tile of adds)

constexpr TsSplit ts_split(int tiles, int units, int nb0, int sms) {
    const bool cut = nb0 == 0 || nb0 >= kTsMinCut;
    int grid = cut ? (units - 1) / kTsMinShare + 1 : tiles;
    // Few tiles: every tile in equally many shares, so that none lies across two tiles and pays for two.  512 x 3584 (four tiles
    // of 28 blocks) with 4 tokens takes 6.3 us in sixteen shares of seven, 7.9 in fourteen of eight, the few-token kernel 6.5; a
    // 7B-shaped W4-G128 layer with 100 tokens, whose pieces are drained one after the other, 133 us after 179.
    if (cut && nb0 > 0) {
        const long long even = (long long)tiles * ((nb0 - 1) / kTsMinShare + 1);
        if (even <= sms) grid = (int)even;
    }
    if (grid > sms) grid = sms;
    TsSplit w = {grid, nb0 > 0 ? tiles / grid : 0, 0, 0, cut ? 1 : nb0};
    w.cut_begin = w.whole * grid * nb0;
    w.cut_units = units - w.cut_begin;
    return w;
}

// Linears of up to 128 tokens that go to the prefill kernel all the same: more tiles than SMs with rows so short that a tile's
// drain, by four warps and above 64 tokens with no second accumulator, takes longer than its blocks; the prefill kernel drains
// with eight.  K = 2, us here and there: 20480 x 1024 (8 blocks) with 128 tokens 17.7 and 12.4, with 72 tokens 14.0 and 11.3; 20480 x 256 with
// 56 tokens 8.8 and 5.0, with 17 tokens 7.3 and 4.5.  Between 3 and 8 blocks below 64 tokens and between 9 and 15 above either may be
// the faster one, by a sixth at most.
constexpr bool ts_drain_bound(int tiles, int nblocks, int M, int sms) {
    return tiles > sms && M > 16 && nblocks <= (M > 64 ? 8 : 2);
}

// Prefill kernel: the stage of a 128-column block (of four 32-column or two 64-column ones) behind which a decode group gives the
// block's packed slot back.  A refill does not queue behind loads that are still out, so every loaded word has to have gone into
// a stored stage: column word q is put together from physical words q and q - 1 (mod 4), so the stage that holds word 2 is the
// first by which all four are used; it also builds the tables of the second coefficient group of g = 64.
constexpr int wide_release_stage(int stages_per_block) { return stages_per_block / 2; }

}  // namespace bpdq
