// tc_skinny.cuh -- skinny tcgen05 contractions (the adapter rank on N) whose
// tiles are few: each 128-row tile belongs to a cluster of CTAs that share its
// K blocks and sum their accumulators through distributed shared memory.
//
// Such a contraction streams a few hundred KB per SM; what it costs is the
// chain of round trips.  The stream-K grouped kernel (tc_group.cuh) ends a
// split tile with partials in global memory, a fence, a ticket, and one CTA
// that reads every other CTA's partial; here the pieces of a tile meet in a
// cluster barrier and every CTA sums its share of the columns, in CTA order
// (the result does not depend on timing).  The adapters are read in place
// (K-major B [r, dout] as rows of a tile, A [din, r] as an MN-major tile of
// half-used 64-column boxes, zero-filled past r), so no kernel has to prepare
// them; only A of a rank that is not a multiple of 8 (TMA cannot read its rows)
// is transposed first.
//
// Measured on GB300 (device time of a call in a replayed graph, grouped form
// against this one): gradients of q and v of the 7B-class update (2,048 rows, r
// 16) 27.9 -> 22.4 us (issued one by one 31.1 -> 24.8), of one 3,584-wide
// projection at 403 rows 19.6 -> 12.4, of four (3,584, 512, 512, 3,584) at 411
// rows, r 32, 53.3 -> 19.3.
// What is left is round trips: setup 0.4 us, first tile 1.3, the K blocks of a
// CTA at 0.2-0.3 each, barrier 0.8, sum and stores 1.3, barrier 0.9.
//
// A tile is a list of segments laid end to end along K, each with its own A
// and B operands and its own accumulator columns: the u and every v_p of a row
// tile in the first pass, one segment in the others.  The i-th of the c CTAs
// that share a tile takes the K blocks [kb[i], kb[i + 1]) of the list, about the
// same cost each (skinny_split).
#pragma once

#include "tc_gemm.cuh"
#include "tc_group.cuh"

namespace attt {

constexpr int kSkinnyThreads = 192;  // producer, MMA, four epilogue warps
constexpr int kSkinnySegs = kMaxProj + 1;
constexpr int kSkinnyMaxCluster = 8;
constexpr int kSkinnyMaxStages = 12;  // ring slots (barriers) of a CTA

struct SkinnySeg {
    int a, b;     // tensor maps: the A operand, the first of nb B operands
    int nb, n;    // B operands sharing the A block, columns of each (a multiple of 16)
    int b_mn;     // B operands MN-major (else K-major)
    int b_n_off;  // first row of a K-major B
    int kb;       // 64-deep K blocks
    int col;      // first accumulator column
    int N;        // columns stored
    int out;      // GroupOut
    float alpha;
    int r, rpad;
    int64_t ld;
    float *out32;
    __nv_bfloat16 *out16;
    float *outp[kMaxProj];
};

// Tiles of M rows in all, each the segments [seg0, seg0 + nseg), on the
// clusters from cluster_begin; `split` CTAs share a tile (a cluster of C holds
// C / split tiles).
struct SkinnyGroup {
    int cluster_begin, split, seg0, nseg, M, ncols;
    int kb[kSkinnyMaxCluster + 1];  // first K block of each of the `split` CTAs, then the total
};

struct SkinnyMaps {
    CUtensorMap a[kSkinnySegs];
    CUtensorMap b[2 * kMaxProj];
};

struct SkinnyArgs {
    int ngroup, nmaps_a, nmaps_b, cluster;
    uint32_t ring_bytes, tmem_cols;
    int *status;
    unsigned int *zero;  // words set to zero (a later launch's counters), or nullptr
    int nzero;
    SkinnyGroup grp[kSkinnySegs];
    SkinnySeg seg[kSkinnySegs];
};

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(addr)
                 : "memory");
    return v;
}

// Sums the column quads [qd, qe) of this thread's row over the nc <= J CTAs
// whose partials start (at this row) at cb[0..nc), in that order, and hands
// each to store(column, sum): U J loads in flight, no division and no look into
// the kernel's parameters per quad (with those, one quad took 0.45 us and the
// 48 of a 192-column tile 22 us of a 69 us pass).
template <int U, int J, class Store>
__device__ __forceinline__ void skinny_sum(int qd, int qe, int nc, const uint32_t (&cb)[kSkinnyMaxCluster],
                                           Store &&store) {
    for (; qd < qe; qd += U) {
        float4 f[U][J];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int j = 0; j < J; ++j)
                f[u][j] = j < nc && qd + u < qe ? ld_cluster_f4(cb[j] + (uint32_t)(qd + u) * 2048u)
                                                : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
            float4 t = f[u][0];
#pragma unroll
            for (int j = 1; j < J; ++j)
                if (j < nc) { t.x += f[u][j].x; t.y += f[u][j].y; t.z += f[u][j].z; t.w += f[u][j].w; }
            if (qd + u < qe) store(4 * (qd + u), t);
        }
    }
}

template <class Store>
__device__ __forceinline__ void skinny_sum_any(int qd, int qe, int nc, const uint32_t (&cb)[kSkinnyMaxCluster],
                                               Store &&store) {
    if (nc <= 2) skinny_sum<8, 2>(qd, qe, nc, cb, store);
    else if (nc <= 4) skinny_sum<4, 4>(qd, qe, nc, cb, store);
    else skinny_sum<2, 8>(qd, qe, nc, cb, store);
}

template <bool A_MN>
__global__ void __launch_bounds__(kSkinnyThreads, 1)
    tc_skinny_kernel(const __grid_constant__ SkinnyMaps maps, const __grid_constant__ SkinnyArgs g) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t ring = smem_u32(smem);  // later the CTA's partial accumulators
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem + g.ring_bytes);
    const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + kSkinnyMaxStages),
                   done = smem_u32(bars + 2 * kSkinnyMaxStages);
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 2 * kSkinnyMaxStages + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    const int rank = g.cluster > 1 ? (int)cluster_ctarank() : 0;
    const int cid = blockIdx.x / g.cluster;
    int q = 0;
    while (q + 1 < g.ngroup && cid >= g.grp[q + 1].cluster_begin) ++q;
    const SkinnyGroup &gr = g.grp[q];
    const int C = gr.split, first = rank - rank % C, part = rank % C;  // the CTAs that share this tile
    const int m0 = ((cid - gr.cluster_begin) * (g.cluster / C) + first / C) * 128;
    const int seg0 = gr.seg0, seg1 = gr.seg0 + gr.nseg;
    const int k0 = gr.kb[part], k1 = m0 < gr.M ? gr.kb[part + 1] : k0;
    // the ring: slots of the largest block this CTA loads, as many as fit (blocks
    // from HBM take 1.5 us and more: five slots hold a CTA to 0.3 us a block)
    uint32_t stage_bytes = kABytes;
    for (int si = seg0, base = 0; si < seg1; base += g.seg[si++].kb) {
        const SkinnySeg &s = g.seg[si];
        if (max(k0, base) < min(k1, base + s.kb))
            stage_bytes = max(stage_bytes, kABytes + (uint32_t)s.nb * (s.b_mn ? 8192u : (uint32_t)s.n * 128u));
    }
    const int S = min(kSkinnyMaxStages, (int)(g.ring_bytes / stage_bytes));

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full0 + 8 * s, 1);
            mbar_init(empty0 + 8 * s, 1);
        }
        mbar_init(done, 1);
        griddep_launch_dependents();
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), g.tmem_cols);
        tmem_relinquish();
    }
    if (warp == 2) {
        for (int i = lane; i < g.nmaps_a + g.nmaps_b; i += 32)
            tma_prefetch_desc(i < g.nmaps_a ? &maps.a[i] : &maps.b[i - g.nmaps_a]);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;

    if (warp == 0) {
        if (elect_one()) {
            griddep_wait();  // the operands may come from the previous grid
            int slot = 0, base = 0, pos = 0;
            uint32_t phase = 1;
            bool ok = true;
            for (int si = seg0; ok && si < seg1; ++si) {
                const SkinnySeg &s = g.seg[si];
                const int kb = s.kb, nb = s.nb, b_mn = s.b_mn, boff = s.b_n_off;
                const uint32_t bytes = kABytes + (uint32_t)nb * (b_mn ? 8192u : (uint32_t)s.n * 128u);
                const CUtensorMap *ta = &maps.a[s.a], *tb = &maps.b[s.b];
                const int ks = max(k0, base) - base, ke = min(k1, base + kb) - base;
                base += kb;
                for (int k = ks; k < ke; ++k, ++pos) {
                    const uint32_t fb = full0 + 8 * slot;
                    if (pos >= S && !mbar_wait(empty0 + 8 * slot, phase, abort_flag)) {
                        ok = false;
                        break;
                    }
                    const uint32_t a_dst = ring + (uint32_t)slot * stage_bytes;
                    mbar_arrive_expect_tx(fb, bytes);
                    if (!A_MN) {
                        tma_load_2d(a_dst, ta, fb, k * 64, m0);
                    } else {
                        tma_load_2d(a_dst, ta, fb, m0, k * 64);
                        tma_load_2d(a_dst + 8192, ta, fb, m0 + 64, k * 64);
                    }
                    if (b_mn) {
                        for (int i = 0; i < nb; ++i) tma_load_2d(a_dst + kABytes + 8192u * i, tb + i, fb, 0, k * 64);
                    } else {
                        tma_load_2d(a_dst + kABytes, tb, fb, k * 64, boff);
                    }
                    if (++slot == S) {
                        slot = 0;
                        phase ^= 1u;
                    }
                }
            }
            if (!ok) {
                *abort_flag = 1;
                record_error(g.status, ATTT_ERR_TIMEOUT);
                // the loads already issued still land in shared memory: wait (bounded, a
                // flag of its own) for each slot's last one
                volatile int no_abort = 0;
                for (int p = pos > S ? pos - S : 0; p < pos; ++p)
                    (void)mbar_wait(full0 + 8 * (p % S), (uint32_t)(p / S) & 1u, &no_abort);
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {
            int slot = 0, base = 0;
            uint32_t phase = 0;
            bool ok = true, ready = false;
            for (int si = seg0; ok && si < seg1; ++si) {
                const SkinnySeg &s = g.seg[si];
                const int kb = s.kb, nb = s.nb, n = s.n;
                const bool b_mn = s.b_mn != 0;
                const uint32_t idesc = idesc_bf16_f32((uint32_t)n, A_MN, b_mn);
                const uint32_t d0 = tmem_base + (uint32_t)s.col;
                const uint32_t b_step = (b_mn ? 2048u : 32u) >> 4;  // a step of 16 along K, in descriptor units
                const int ks = max(k0, base) - base, ke = min(k1, base + kb) - base;
                base += kb;
                for (int k = ks; k < ke; ++k) {
                    if (!ready && !mbar_wait(full0 + 8 * slot, phase, abort_flag)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    // the next slot's barrier is read while this slot's MMAs issue
                    const int next = slot + 1 == S ? 0 : slot + 1;
                    const uint32_t next_phase = next == 0 ? phase ^ 1u : phase;
                    ready = mbar_test_wait(full0 + 8 * next, next_phase);
                    const uint32_t a_addr = ring + (uint32_t)slot * stage_bytes;
                    const uint64_t ad = smem_desc_sw128(a_addr, A_MN ? 8192 : 16, 1024);
                    for (int i = 0; i < nb; ++i) {
                        const uint64_t bd = smem_desc_sw128(a_addr + kABytes + 8192u * i, b_mn ? 8192 : 16, 1024);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            umma_bf16(d0 + (uint32_t)(i * n), ad + kk * ((A_MN ? 2048u : 32u) >> 4), bd + kk * b_step,
                                      idesc, (k > ks || kk > 0) ? 1u : 0u);
                    }
                    umma_commit(empty0 + 8 * slot);
                    slot = next;
                    phase = next_phase;
                }
            }
            if (!ok) {
                *abort_flag = 1;
                record_error(g.status, ATTT_ERR_TIMEOUT);
                // The producer may have issued every load and gone: those that no MMA
                // waited for (at most a ring of them) land before the CTA retires, as far
                // as bounded waits of this thread's own can see to it.
                volatile int no_abort = 0;
                for (int i = 0; i < S && mbar_wait(full0 + 8 * slot, phase, &no_abort); ++i)
                    if (++slot == S) {
                        slot = 0;
                        phase ^= 1u;
                    }
            }
            umma_commit(done);
        }
        __syncwarp();
    }

    // Every issued MMA has completed (bounded wait) before its accumulators are
    // read or freed, and with them every load of the ring.
    {
        volatile int no_abort = 0;
        int ok = 1;
        if (lane == 0) ok = mbar_wait(done, 0u, &no_abort) ? 1 : 0;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        if (!ok && lane == 0) record_error(g.status, ATTT_ERR_TIMEOUT);
        if (ok) (void)mbar_try_wait(done, 0u);
        tc_fence_after();
    }

    const int row = (warp & 3) * 32 + lane;  // epilogue warps 2..5: quarters 2, 3, 0, 1
    if (warp >= 2) {
        if (blockIdx.x == 0 && g.zero) {
            griddep_wait();
            for (int i = threadIdx.x - 64; i < g.nzero; i += 128) g.zero[i] = 0u;
        }
        const uint32_t taddr = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
        int base = 0;
        for (int si = seg0; si < seg1; base += g.seg[si++].kb) {
            const SkinnySeg &s = g.seg[si];
            if (max(k0, base) >= min(k1, base + s.kb)) continue;  // not this CTA's
            for (int c = s.col; c < s.col + s.nb * s.n; c += 16) {
                float v[16];
                tmem_ld_x16(taddr + (uint32_t)c, v);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    st_shared_f4(ring + (uint32_t)((c / 4 + j) * 128 + row) * 16u,
                                 make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
            }
        }
        tc_fence_before();
    }
    if (g.cluster > 1) cluster_sync();  // every CTA's partials are in its shared memory
    else __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, g.tmem_cols);
    }
    if (warp >= 2 && m0 < gr.M) {
        const int m = m0 + row;
        const int nq = gr.ncols / 4, q1 = nq * (part + 1) / C;
        int base = 0;
        for (int si = seg0; si < seg1; base += g.seg[si++].kb) {
            const SkinnySeg &s = g.seg[si];
            // the quads of columns of this segment in this CTA's share, and the CTAs
            // [c0, c0 + nc) that hold K blocks of it
            int qd = max(nq * part / C, s.col / 4);
            const int qe = min(q1, (s.col + s.nb * s.n) / 4);
            if (qd >= qe) continue;
            int c0 = 0, nc = 0;
            for (int j = 0; j < C; ++j)
                if (max(gr.kb[j], base) < min(gr.kb[j + 1], base + s.kb)) {
                    if (nc == 0) c0 = j;
                    ++nc;
                }
            uint32_t cb[kSkinnyMaxCluster];
#pragma unroll
            for (int j = 0; j < kSkinnyMaxCluster; ++j)
                cb[j] = mapa_shared(ring + (uint32_t)row * 16u, (uint32_t)(first + min(c0 + j, C - 1)));
            // the sums' columns are the tile's; the segment's start at col.  Rows past
            // the problem are summed (the loads are harmless) and not stored.
            const int col = s.col, N = s.N, r = s.r;
            const bool live = m < gr.M;
            const float al = s.alpha;
            const int64_t ld = s.ld;
            if (s.out == GOUT_T16) {
                __nv_bfloat16 *o = s.out16 + m - (int64_t)col * ld;
                skinny_sum_any(qd, qe, nc, cb, [&](int n, const float4 &t) {
                    const float v[4] = {al * t.x, al * t.y, al * t.z, al * t.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (live && n + i - col < N) o[(int64_t)(n + i) * ld] = __float2bfloat16_rn(v[i]);
                });
            } else if (s.out == GOUT_N32) {
                // projection by projection: a block of rpad columns each
                const int rpad = s.rpad;
                for (int blk = (4 * qd - col) / rpad; qd < qe; ++blk) {
                    const int be = min(qe, (col + (blk + 1) * rpad) / 4), c0b = col + blk * rpad;
                    float *o = s.outp[blk] + (int64_t)m * r;
                    const bool vec = (r & 3) == 0 && (reinterpret_cast<uintptr_t>(s.outp[blk]) & 15) == 0;
                    skinny_sum_any(qd, be, nc, cb, [&](int n, const float4 &t) {
                        const float v[4] = {al * t.x, al * t.y, al * t.z, al * t.w};
                        const int c = n - c0b;
                        if (live && vec && c + 4 <= r) {
                            *reinterpret_cast<float4 *>(o + c) = make_float4(v[0], v[1], v[2], v[3]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 4; ++i)
                                if (live && c + i < r) o[c + i] = v[i];
                        }
                    });
                    qd = be;
                }
            } else if (s.out == GOUT_T32) {
                float *o = s.out32 + m - (int64_t)col * ld;
                skinny_sum_any(qd, qe, nc, cb, [&](int n, const float4 &t) {
                    const float v[4] = {al * t.x, al * t.y, al * t.z, al * t.w};
#pragma unroll
                    for (int i = 0; i < 4; ++i)
                        if (live && n + i - col < r) o[(int64_t)(n + i) * ld] = v[i];
                });
            } else {  // GOUT_N16: ld a multiple of 16, the base 256-byte aligned
                __nv_bfloat16 *o = s.out16 + (int64_t)m * ld - col;
                skinny_sum_any(qd, qe, nc, cb, [&](int n, const float4 &t) {
                    __nv_bfloat162 b[2] = {__floats2bfloat162_rn(al * t.x, al * t.y),
                                           __floats2bfloat162_rn(al * t.z, al * t.w)};
                    if (live) *reinterpret_cast<uint2 *>(o + n) = *reinterpret_cast<uint2 *>(b);
                });
            }
        }
    }
    if (g.cluster > 1) cluster_sync();  // no CTA leaves while another reads its partials
}

}  // namespace attt
