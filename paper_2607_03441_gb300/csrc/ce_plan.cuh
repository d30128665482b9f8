// ce_plan.cuh -- how an Eq. 10 call (ce.cu) is cut: the width of its vocabulary
// chunks and the tiles of its two contractions.  Host code.
#pragma once

#include "gemm_launch.cuh"

namespace attt {

constexpr int kCeBN = 256;
// (max, sum) pairs of sets narrower than those of 256-column tiles, at most: the
// plan takes narrow tiles only where few tiles would leave SMs idle (L 1 to
// 20,000, V 256 to 262,144, d 64 to 8,192 on 152 SMs: at most 1,125,316 pairs).
constexpr int64_t kCeNarrowPairs = 5ll << 18;  // 10 MB
constexpr int kCeMaxTiles = 1024;  // chunk width at most, in kCeBN columns
static_assert(kCeMaxTiles * kCeBN <= kCeMaxChunk, "the fp32 range of dh is argued for chunks of kCeMaxChunk columns");
// Bound of the chunk's bf16 block E [L, Vc] in bytes.
constexpr int64_t kCeEBytes = 1024ll << 20;
// Columns that one fp32 accumulation of dh runs over, at most: the tensor core's
// sums lose a little with their length.  Error of dh against 64 bits at L 2,048, d
// 3,584, three seeds: 6.21e-4 in chains of 50,688 columns, 6.34e-4 in one of
// 152,064 (the bf16 rounding of E is nearly all of both).  A chunk may be wider
// where K pieces cut the chain.
constexpr int64_t kCeMaxChain = 65536;
// dh tiles of 256 x 256 above which a chunk never runs in K pieces (76 CTA pairs
// and 160 regions of partials), so that its width is bounded by kCeMaxChain.
constexpr int64_t kCeWholeTiles = 64;

// Upper bound of the vocab chunk: the chunk's bf16 block E (L x Vc) is kept
// near kCeEBytes (1 GB), so the workspace stays bounded whatever V is.  Each
// chunk costs about 20 us of launch, ramp and tail on top of its FLOPs, and E is streamed
// once from L2 or HBM either way, so wider chunks are faster up to this bound
// (d 3,584, V 152,064, calls back to back, one chunk against three: L 93 350
// against 391 us, L 403 698 against 768; L 2,048, where the chain is bounded,
// would take 2,640 against 2,670 at the power cap, and a workspace of 675
// instead of 321 MB).
inline int64_t ce_chunk_max(int64_t L, int64_t d, int64_t V) {
    int64_t vc = kCeEBytes / (2 * L);
    vc = (vc / kCeBN) * kCeBN;
    if (vc < 4096) vc = 4096;
    const int64_t most = cdiv(L, 256) * cdiv(d, 256) > kCeWholeTiles ? kCeMaxChain : (int64_t)kCeMaxTiles * kCeBN;
    if (vc > most) vc = most;
    const int64_t vmax = round_up(V, kCeBN);
    if (vc > vmax) vc = vmax;
    return vc;
}

// Chunk width and the tiles of both contractions for `sms` SMs.
struct CePlan {
    int64_t Vc;
    TilePlan logits, dh;
};

// Epilogue sets of a logits tile.
inline int ce_sets(int64_t d) { return cdiv(d, 64) <= kTwoSetBlocks ? 2 : 1; }

// (max, sum) pairs that the sets of a chunk of Vc columns may need.
inline int64_t ce_pairs(int64_t L, int64_t d, int64_t Vc) {
    const int64_t wide = cdiv(Vc, kCeBN) * ce_sets(d) * L, most = cdiv(Vc, 64) * ce_sets(d) * L;
    const int64_t narrow = most < kCeNarrowPairs ? most : kCeNarrowPairs;
    return wide > narrow ? wide : narrow;
}

inline CePlan ce_plan(int64_t L, int64_t d, int64_t V, int regions, int sms) {
    CePlan p{};
    const int64_t vmax = ce_chunk_max(L, d, V);
    for (int64_t n = cdiv(V, vmax);; ++n) {  // the fewest equal chunks that keep the chains short
        p.Vc = round_up(cdiv(V, n), kCeBN);
        p.dh = plan_tiles(L, d, cdiv(p.Vc, 64), sms, regions, true, true);
        if (cdiv(cdiv(p.Vc, 64), p.dh.pieces) * 64 <= kCeMaxChain) break;
    }
    p.logits = plan_tiles(L, p.Vc, cdiv(d, 64), sms, 0, false, false);
    const int64_t pairs = ce_pairs(L, d, vmax);
    while (p.logits.BN < kCeBN && cdiv(p.Vc, p.logits.BN / ce_sets(d)) * L > pairs) p.logits.BN += 64;
    return p;
}

}  // namespace attt
