// gemm_launch.cuh -- host-side set-up and launch of tc_gemm_kernel.
#pragma once

#include "attt_host.h"
#include "tc_gemm.cuh"

namespace attt {

// Description of one contraction D = A * B^T (see tc_gemm.cuh).
struct GemmProblem {
    const void *a;        // A base pointer
    int64_t a_rows_ld;    // A: K-major -> row pitch in elements of the [rows, K] matrix;
                          //    MN-major -> row pitch of the [K, rows] matrix
    int64_t a_rows, a_k;  // extents of A's storage (rows = M extent, k = K extent)
    const void *b;
    int64_t b_rows_ld;
    int64_t b_rows, b_k;
    int M, N, K;
    // optional second operand pair over K2 more K (same majors, no offsets):
    // D = A B^T + A2 B2^T
    const void *a2 = nullptr;
    int64_t a2_rows_ld = 0, a2_rows = 0, a2_k = 0;
    const void *b2 = nullptr;
    int64_t b2_rows_ld = 0, b2_rows = 0, b2_k = 0;
    int K2 = 0;
    int BN;
    int a_m_off = 0, a_k_off = 0, b_n_off = 0, b_k_off = 0;
    bool pair = false;  // run on CTA pairs (256-row tiles, cta_group::2)
    // Launch as a programmatic dependent of the previous grid in the stream;
    // operands_ready: A and B do not come from that grid.
    bool pdl = false;
    bool operands_ready = false;
    bool second_waits = false;  // with operands_ready: A2 and B2 do come from it
    // Tail split (EPI_F32_ACC): workspace for up to `split_regions` partials
    // of 128 x BN fp32 and as many arrival counters (zero on entry).
    float *split_ws = nullptr;
    unsigned int *split_tick = nullptr;
    int split_regions = 0;
    // EPI_F32_PART: K pieces per tile; each stores its 128-row accumulators
    // (pair: 256) at its part_row of split_ws, BN columns wide.
    int pieces = 1;
};

// Pieces per tile for the tiles of a partial last wave: `tiles` tiles over
// `units` concurrent tile slots leave r = tiles mod units tiles for the last
// wave; cutting each into s K pieces (2 <= s <= 4, at least 8 K blocks each)
// runs that wave in ceil(r s / units) / s of a tile's time.  Returns 1 when the
// cut shortens the launch by less than a tenth (a long launch under the power
// cap gains nothing from filling idle SMs) or the partials would not fit
// `regions` (ranks per tile: `nranks`).
inline int tail_pieces(int tiles, int units, int kb_total, int nranks, int regions) {
    const int r = tiles % units;
    if (r == 0) return 1;
    int best_s = 1;
    double best = 1.0;
    for (int s = 2; s <= 4; ++s) {
        if (kb_total < 8 * s || r * s * nranks > regions) break;
        const double t = (double)cdiv(r * s, units) / s;
        if (t < best - 1e-9) { best = t; best_s = s; }
    }
    const double waves = (double)(tiles / units) + 1.0;
    return (1.0 - best) >= 0.1 * waves ? best_s : 1;
}

// Arguments of the kernel that ends an EPI_F32_PART contraction: out (fp32) =
// (accumulate ? alpha_m out : 0) + beta_m sum [- gamma_m W[t_m, :]], as
// EPI_F32_ACC, or out16 (bf16) = alpha sum, as EPI_BF16.  N is a multiple of 4.
struct SplitReduceArgs {
    const float *part;
    int M, N, BN, pieces, rows, tiles_m;  // rows: accumulator rows per tile (128, pair: 256)
    int64_t ld;
    float *out;
    __nv_bfloat16 *out16;
    float alpha;
    int accumulate;
    const float *row_alpha, *row_beta, *row_gamma;
    const int32_t *fix_tgt;
    const __nv_bfloat16 *fix_W;
    int64_t fix_ld;
    int fix_V;
};
attt_status launch_split_reduce(const SplitReduceArgs &a, cudaStream_t stream);

// How a contraction is cut: CTA pairs or single CTAs, the tile width, and the
// K pieces every tile runs as.
struct TilePlan {
    bool pair;
    int BN, pieces;
};

// Constants of the plan's estimate, fitted to Eq. 10 calls on GB300 (L 33 to
// 8,000, every width and both CTA forms): one 64-deep K block takes an SM the
// time of its MMAs or of its operands from L2, whichever is longer.  Measured
// per block: 0.33 us for a 256 x 256 pair tile, 0.22 for 256 x 128; single CTAs
// 0.43-0.47 / 0.35-0.38 / 0.24-0.29 / 0.20 us for the 48 / 40 / 32 / 24 KB of a
// 128 x 256 / 192 / 128 / 64 tile.  Single CTAs and narrow tiles draw more from
// L2 per FLOP, so they pay only where they fill idle SMs.
constexpr int kMaxPieces = 16;
constexpr double kSmFlops = 12.5e12;                       // bf16 FLOP/s of one SM
constexpr double kTileFixed = 3e-6, kTileColumn = 1.2e-8;  // ramp of a launch; epilogue of its last tile
constexpr double kReduceFixed = 3e-6, kReduceByte = 1.6e-13;  // the pieces' reduction (split_reduce.cu)
constexpr double kTailSum = 1.8e-5;                        // the tail split's partials and their sum

// A K block's operands into one SM: 62 bytes a cycle from L2.
inline double block_feed_seconds(bool pair, int BN, bool b_mn) {
    const int cols = !pair ? BN : b_mn ? (int)round_up(BN / 2, 64) : BN / 2;
    return 9e-9 * (16.0 + cols / 8.0);
}

// The plan of least estimated time for an M x N result over kb 64-deep K
// blocks on `sms` SMs.  `regions` bounds the fp32 partials of the K pieces
// (in 128 x 256 blocks; 0: whole tiles); `tail`: the whole-tile form may cut
// the tiles of its last wave (tail_pieces).  MN-major B operands (b_mn) come
// in 64-column boxes, hence the widths.  A width that fills whole waves beats a
// wider one that does not: 2,048 x 3,584 has 112 tiles of 256 columns for 76
// pairs (1.47 waves) and 152 of 192 (2.0).  Cutting pays when the tiles leave SMs
// idle: at 256 rows, d 512, V 8,192 the dh contraction's 2 tiles took 36 us as
// 4 pieces each and take 6 us as 16 of 128 columns; at 93 rows, d 3,584,
// V 152,064 its 14 tiles took 337 us as 4 pieces of 4 chunks and take 170 us
// as 10 pieces of one.
inline TilePlan plan_tiles(int64_t M, int64_t N, int64_t kb, int sms, int64_t regions, bool tail,
                           bool b_mn) {
    TilePlan best{true, 256, 1};
    double best_t = 1e30;
    for (int pair = 1; pair >= 0; --pair) {
        const int64_t rows = pair ? 256 : 128, units = pair ? sms / 2 : sms;
        for (int BN = 256; BN >= 64; BN -= 64) {
            if (pair && BN == 64) continue;
            const int64_t tiles = cdiv(M, rows) * cdiv(N, BN);
            // (pair tiles of 192 columns run their MMAs at 0.29 us a block, not 0.25)
            const double mma = pair && BN == 192 ? 0.29e-6 : 128.0 * BN * 128 / kSmFlops;
            const double feed = block_feed_seconds(pair, BN, b_mn), block = mma > feed ? mma : feed;
            for (int64_t s = 1; s <= kMaxPieces; ++s) {
                if (s > 1 && (kb < 16 * s || tiles * s * (rows / 128) * BN > regions * 256)) break;
                double waves = (double)cdiv(tiles * s, units), extra = 0.0;
                if (s == 1 && tail) {
                    const int cut = tail_pieces((int)tiles, (int)units, (int)kb, (int)(rows / 128), (int)regions);
                    if (cut > 1) {
                        waves = (double)(tiles / units) + (double)cdiv(tiles % units * cut, units) / cut;
                        extra = kTailSum;
                    }
                }
                if (s > 1) extra = kReduceFixed + kReduceByte * 8.0 * s * M * N;
                const double t = waves * cdiv(kb, s) * block + kTileFixed + BN * kTileColumn + extra;
                if (t < 0.98 * best_t) {  // the wider and whole forms at equal estimates
                    best_t = t;
                    best = TilePlan{pair != 0, BN, (int)s};
                }
            }
        }
    }
    return best;
}

// Tile order: with all row tiles walked per column tile, every wave streams
// all of A (a_bytes); once A exceeds half of L2, groups of `group` tiles (2,048
// rows; of rows_tile each) keep theirs there and a wave of 76 pair tiles reads 8
// row and 9.5 column blocks instead of 32 and 2.4.  At 8,192 x 5,120 x
// 152,064 the logits contractions read 2.6 instead of 5.2 GB from DRAM and the dh
// contractions 5.8 instead of 9.7 (per chunk, on one GPU; the concurrent tiles
// drift apart along K, and in five captures the groups read 2.4 to 3.6 and 5.1 to
// 8.7), the call at the power cap 15.9 -> 15.0 ms; where A fits (4,096 x 4,096)
// the logits lose 1% by it.  0: no groups.
inline int tile_group(int64_t M, int rows_tile, int group, double a_bytes) {
    return a_bytes > 64e6 && cdiv(M, rows_tile) > 2 * group ? group : 0;
}

constexpr size_t kMaxSmem = 232448;  // 227 KB opt-in per CTA on sm_100-class parts

inline int gemm_stages(int BN, uint32_t extra = 0) {
    int s = 8;
    while (s > 2 && gemm_smem_bytes(BN, s, extra) > kMaxSmem) --s;
    return s;
}

inline uint32_t gemm_tmem_cols(int BN) {
    uint32_t need = 2u * (uint32_t)BN, c = 32;
    while (c < need) c <<= 1;
    return c;
}

// `status` is the device word that records a timed-out wait; nullptr selects
// the library's per-device status word.
template <int EPI, bool A_MN, bool B_MN, int SETS = 1>
attt_status launch_gemm(const GemmProblem &p, const EpiParams &ep, int dev, cudaStream_t stream,
                        int *status = nullptr) {
    if (p.BN < 16 || p.BN > 256 || p.BN % 16 != 0) return ATTT_ERR_INVALID_ARG;
    if (SETS == 2 && p.BN % 64 != 0) return ATTT_ERR_INVALID_ARG;  // sets of 32-column chunks
    if (B_MN && p.BN % 64 != 0) return ATTT_ERR_INVALID_ARG;
    if (p.pair && p.BN < 32) return ATTT_ERR_INVALID_ARG;  // BN/2 B rows per CTA (a multiple of 8)
    if (p.M <= 0 || p.N <= 0 || p.K <= 0) return ATTT_ERR_INVALID_ARG;
    CUtensorMap ta, tb;
    // K-major operand: storage [rows, K] (K contiguous), box 64 x rows_tile.
    // MN-major operand: storage [K, rows] (rows contiguous), box 64 x 64.
    bool ok;
    // EPI_KL loads 64 rows of A and 64 of A2 into one 128-row tile
    const uint32_t a_box_rows = EPI == EPI_KL ? 64u : 128u;
    if (!A_MN)
        ok = make_tmap_bf16(&ta, p.a, (uint64_t)p.a_k, (uint64_t)p.a_rows, (uint64_t)p.a_rows_ld * 2, 64, a_box_rows);
    else
        ok = make_tmap_bf16(&ta, p.a, (uint64_t)p.a_rows, (uint64_t)p.a_k, (uint64_t)p.a_rows_ld * 2, 64, 64);
    if (!ok) return ATTT_ERR_INVALID_ARG;
    if (!B_MN)
        ok = make_tmap_bf16(&tb, p.b, (uint64_t)p.b_k, (uint64_t)p.b_rows, (uint64_t)p.b_rows_ld * 2, 64,
                            (uint32_t)(p.pair ? p.BN / 2 : p.BN));
    else
        ok = make_tmap_bf16(&tb, p.b, (uint64_t)p.b_rows, (uint64_t)p.b_k, (uint64_t)p.b_rows_ld * 2, 64, 64);
    if (!ok) return ATTT_ERR_INVALID_ARG;
    CUtensorMap ta2 = ta, tb2 = tb;
    if (EPI == EPI_KL) {
        // the second A operand (same shape as A) shares every B tile
        if (!p.a2 || !p.pair || A_MN || B_MN) return ATTT_ERR_INVALID_ARG;
        if (!make_tmap_bf16(&ta2, p.a2, (uint64_t)p.a_k, (uint64_t)p.a_rows, (uint64_t)p.a2_rows_ld * 2, 64, 64))
            return ATTT_ERR_INVALID_ARG;
    } else if (p.K2 > 0) {
        if (!p.a2 || !p.b2) return ATTT_ERR_INVALID_ARG;
        if (!A_MN)
            ok = make_tmap_bf16(&ta2, p.a2, (uint64_t)p.a2_k, (uint64_t)p.a2_rows, (uint64_t)p.a2_rows_ld * 2, 64, 128);
        else
            ok = make_tmap_bf16(&ta2, p.a2, (uint64_t)p.a2_rows, (uint64_t)p.a2_k, (uint64_t)p.a2_rows_ld * 2, 64, 64);
        if (!ok) return ATTT_ERR_INVALID_ARG;
        if (!B_MN)
            ok = make_tmap_bf16(&tb2, p.b2, (uint64_t)p.b2_k, (uint64_t)p.b2_rows, (uint64_t)p.b2_rows_ld * 2, 64,
                                (uint32_t)(p.pair ? p.BN / 2 : p.BN));
        else
            ok = make_tmap_bf16(&tb2, p.b2, (uint64_t)p.b2_rows, (uint64_t)p.b2_k, (uint64_t)p.b2_rows_ld * 2, 64, 64);
        if (!ok) return ATTT_ERR_INVALID_ARG;
    }
    // EPI_CE_EXP writes E through TMA stores: [M, G_ld] bf16, 32 x 32 boxes
    // EPI_F32_ACC reads and writes `out` through TMA: [M, N] fp32 of pitch out_ld, 32 x 32 boxes
    CUtensorMap tc = tb;
    if (EPI == EPI_CE_EXP) {
        if (!make_tmap_bf16(&tc, ep.G, (uint64_t)ep.G_ld, (uint64_t)p.M, (uint64_t)ep.G_ld * 2, 32, 32, 64))
            return ATTT_ERR_INVALID_ARG;
    } else if (EPI == EPI_F32_ACC) {
        if (!make_tmap_f32(&tc, ep.out, (uint64_t)p.N, (uint64_t)p.M, (uint64_t)ep.out_ld * 4, 32, 32))
            return ATTT_ERR_INVALID_ARG;
    } else if (EPI == EPI_F32_PART) {
        const int64_t t = cdiv(p.M, p.pair ? 256 : 128) * cdiv(p.N, p.BN) * p.pieces * (p.pair ? 2 : 1);
        if (!p.split_ws || p.pieces < 1 || t * p.BN > (int64_t)p.split_regions * 256) return ATTT_ERR_INVALID_ARG;
        if (!make_tmap_f32(&tc, p.split_ws, (uint64_t)p.BN, (uint64_t)t * 128, (uint64_t)p.BN * 4, 32, 32))
            return ATTT_ERR_INVALID_ARG;
    } else if (EPI == EPI_BF16) {
        if (!make_tmap_bf16(&tc, ep.out16, (uint64_t)p.N, (uint64_t)p.M, (uint64_t)ep.out_ld * 2, 32, 32, 64))
            return ATTT_ERR_INVALID_ARG;
    }

    GemmArgs g{};
    g.M = p.M;
    g.N = p.N;
    g.BN = p.BN;
    // B rows one CTA stages (whole 64-column boxes when MN-major)
    const int bn_cta = !p.pair ? p.BN : B_MN ? (int)round_up(p.BN / 2, 64) : p.BN / 2;
    g.e_stage_bytes = (EPI == EPI_CE_EXP || EPI == EPI_BF16) ? SETS * kEStageBytes
                      : (EPI == EPI_F32_ACC || EPI == EPI_F32_PART) ? kF32StageBytes
                      : EPI == EPI_KL                        ? kKlXBytes
                                                             : 0u;
    g.stages = gemm_stages(bn_cta, g.e_stage_bytes);
    // tiles_m counts tiles of 128 accumulator rows; an EPI_KL tile holds 64
    // rows of the problem (the other 64 are A2's)
    g.tiles_m = (int)cdiv(p.M, EPI == EPI_KL ? 64 : 128);
    g.tiles_n = (int)cdiv(p.N, p.BN);
    g.kb_split = (int)cdiv(p.K, 64);
    g.kb_total = g.kb_split + (p.K2 > 0 ? (int)cdiv(p.K2, 64) : 0);
    const int sms = num_sms(dev);
    const int units = p.pair ? sms / 2 : sms;  // concurrent tiles
    const int tiles = (p.pair ? (g.tiles_m + 1) / 2 : g.tiles_m) * g.tiles_n;
    g.splits = 1;
    g.kb_per_split = g.kb_total;
    g.whole_tiles = tiles;
    g.tail_s = 1;
    if (EPI == EPI_F32_PART) {
        g.whole_tiles = 0;
        g.tail_s = p.pieces;
    }
    if (EPI == EPI_F32_ACC && p.split_ws && p.split_tick && p.BN % 32 == 0) {
        const int s = tail_pieces(tiles, units, g.kb_total, p.pair ? 2 : 1, p.split_regions);
        if (s > 1) {
            g.tail_s = s;
            g.whole_tiles = tiles - tiles % units;
            g.split_ws = p.split_ws;
            g.split_tick = p.split_tick;
        }
    }
    g.a_m_off = p.a_m_off;
    g.a_k_off = p.a_k_off;
    g.b_n_off = p.b_n_off;
    g.b_k_off = p.b_k_off;
    g.tmem_cols = gemm_tmem_cols(p.BN);
    g.operands_ready = !p.operands_ready ? 0 : p.second_waits ? 2 : 1;
    const int rows_tile = EPI == EPI_KL ? 128 : p.pair ? 256 : 128;
    const int group = EPI == EPI_KL ? 8 : 2048 / rows_tile;
    g.group_m = tile_group(p.M, rows_tile, group, 2.0 * p.M * p.K * (EPI == EPI_KL ? 2 : 1));
    g.status = status ? status : device_status_word(dev);
    g.ep = ep;

    const size_t smem = gemm_smem_bytes(bn_cta, g.stages, g.e_stage_bytes);
    const int ntiles = g.whole_tiles + (tiles - g.whole_tiles) * g.tail_s;  // work items
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3((unsigned)(p.pair ? gemm_pair_threads(SETS) : gemm_threads(SETS)));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    unsigned na = 0;
    if (p.pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    if (!p.pair) {
        if constexpr (EPI != EPI_KL) {  // EPI_KL runs on CTA pairs only
            auto kern = tc_gemm_kernel<EPI, A_MN, B_MN, SETS>;
            if (!set_smem_limit(reinterpret_cast<const void *>(kern), smem, dev)) return ATTT_ERR_CUDA;
            cfg.gridDim = dim3((unsigned)(ntiles < sms ? ntiles : sms));
            cfg.attrs = attr;
            cfg.numAttrs = na;
            if (cudaLaunchKernelEx(&cfg, kern, ta, tb, tc, ta2, tb2, g) != cudaSuccess) return ATTT_ERR_CUDA;
        }
    } else {
        auto kern = tc_gemm_pair_kernel<EPI, A_MN, B_MN, SETS>;
        if (!set_smem_limit(reinterpret_cast<const void *>(kern), smem, dev)) return ATTT_ERR_CUDA;
        const int pairs = ntiles < units ? ntiles : units;
        cfg.gridDim = dim3((unsigned)(2 * pairs));
        attr[na].id = cudaLaunchAttributeClusterDimension;
        attr[na].val.clusterDim.x = 2;
        attr[na].val.clusterDim.y = 1;
        attr[na].val.clusterDim.z = 1;
        ++na;
        cfg.attrs = attr;
        cfg.numAttrs = na;
        if (cudaLaunchKernelEx(&cfg, kern, ta, tb, tc, ta2, tb2, g) != cudaSuccess) return ATTT_ERR_CUDA;
    }
    count_launch();
    return cudaGetLastError() == cudaSuccess ? ATTT_OK : ATTT_ERR_CUDA;
}

// A contraction with an fp32 (ep.out) or bf16 (ep.out16) result on the tiles of
// `t`: whole tiles with the fused epilogue, or K pieces and the reduction.
template <bool OUT16, bool A_MN, bool B_MN>
attt_status launch_planned(GemmProblem p, const EpiParams &ep, const TilePlan &t, int dev, cudaStream_t stream) {
    p.pair = t.pair;
    p.BN = t.BN;
    if (t.pieces == 1) return launch_gemm<OUT16 ? EPI_BF16 : EPI_F32_ACC, A_MN, B_MN>(p, ep, dev, stream);
    p.pieces = t.pieces;
    const attt_status st = launch_gemm<EPI_F32_PART, A_MN, B_MN>(p, ep, dev, stream);
    if (st != ATTT_OK) return st;
    SplitReduceArgs a{};
    a.part = p.split_ws;
    a.M = p.M; a.N = p.N; a.BN = t.BN; a.pieces = t.pieces; a.rows = t.pair ? 256 : 128;
    a.tiles_m = (int)cdiv(p.M, a.rows);
    a.ld = ep.out_ld; a.alpha = ep.alpha;
    if (OUT16) a.out16 = ep.out16;
    else a.out = ep.out;
    a.accumulate = ep.accumulate;
    a.row_alpha = ep.row_alpha; a.row_beta = ep.row_beta; a.row_gamma = ep.row_gamma;
    a.fix_tgt = ep.fix_tgt; a.fix_W = ep.fix_W; a.fix_ld = ep.fix_ld; a.fix_V = ep.fix_V;
    return launch_split_reduce(a, stream);
}

}  // namespace attt
