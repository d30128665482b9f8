"""The host side of the tile plans and of the tile order, compiled from the
library's own headers: every K piece is stored where the kernel that sums the
pieces reads it, and the plan of Eq. 10 keeps its bounds."""
import subprocess

import pytest

from paper_2607_03441_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "ce_plan.cuh"
using namespace attt;

// One planned contraction, M x N over K, as launch_planned and launch_gemm cut
// and order it; prints: pieces, group, column tiles, pieces that are not where
// the sum looks for them (or past the regions, or stored twice).
static void walk(int64_t M, int64_t N, int64_t K, int64_t K2, int regions, bool tail, bool b_mn) {
    const int64_t kb = cdiv(K, 64) + cdiv(K2, 64);
    const TilePlan t = plan_tiles(M, N, kb, 152, regions, tail, b_mn);
    const int rows = t.pair ? 256 : 128, tiles_m = (int)cdiv(M, rows);
    GemmArgs g{};
    g.tiles_n = (int)cdiv(N, t.BN);
    g.kb_total = (int)kb;
    g.group_m = tile_group(M, rows, 2048 / rows, 2.0 * M * K);
    g.whole_tiles = t.pieces > 1 ? 0 : tiles_m * g.tiles_n;
    g.tail_s = t.pieces;
    const int nwork = work_count(g, tiles_m);
    int bad = 0;
    if (t.pieces > 1) {
        std::vector<long> owner((size_t)nwork, -1);  // of each region: the (tile, piece) stored there
        for (int w = 0; w < nwork; ++w) {
            const Work k = work_item(g, w, tiles_m);
            const int64_t y = part_row(k.tm, k.tn, tiles_m, k.piece, t.pieces, rows);
            if (y % rows || y < 0 || y / rows >= nwork || owner[y / rows] != -1 || k.kb0 >= k.kb1) ++bad;
            else owner[y / rows] = ((long)k.tn * tiles_m + k.tm) * t.pieces + k.piece;
        }
        for (int64_t row = 0; row < M; row += rows)  // as split_reduce_kernel finds them
            for (int64_t col = 0; col < N; col += t.BN)
                for (int p = 0; p < t.pieces; ++p) {
                    const int64_t y = part_row((int)(row / rows), (int)(col / t.BN), tiles_m, 0, t.pieces, rows);
                    const long want = ((long)(col / t.BN) * tiles_m + row / rows) * t.pieces + p;
                    if (owner[y / rows + p] != want) ++bad;
                }
        if ((int64_t)nwork * rows * t.BN > (int64_t)regions * 128 * 256) ++bad;
    }
    std::printf("%d %d %d %d\n", t.pieces, g.group_m, g.tiles_n, bad);
}

// The plan of an Eq. 10 call: chunk width and its bound, columns of the longest
// accumulation of dh, (max, sum) pairs and the pairs there is room for.
static void eq10(int64_t L, int64_t d, int64_t V, int regions, int sms) {
    const CePlan p = ce_plan(L, d, V, regions, sms);
    std::printf("%lld %lld %lld %lld %lld\n", (long long)p.Vc, (long long)ce_chunk_max(L, d, V),
                (long long)(cdiv(cdiv(p.Vc, 64), p.dh.pieces) * 64),
                (long long)(cdiv(p.Vc, p.logits.BN / ce_sets(d)) * L), (long long)ce_pairs(L, d, ce_chunk_max(L, d, V)));
}

int main(int argc, char **) {
    long long M, N, K, K2;
    int regions, tail, b_mn;
    if (argc > 1)
        while (std::scanf("%lld %lld %lld %d %d", &M, &N, &K, &regions, &tail) == 5) eq10(M, N, K, regions, tail);
    else
        while (std::scanf("%lld %lld %lld %lld %d %d %d", &M, &N, &K, &K2, &regions, &tail, &b_mn) == 7)
            walk(M, N, K, K2, regions, tail != 0, b_mn != 0);
}
"""


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    src, exe = d / "walk.cu", d / "walk"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, str(src), "-o", str(exe)], check=True)

    def run(shapes, *args):
        text = "\n".join(" ".join(str(int(v)) for v in s) for s in shapes)
        out = subprocess.run([str(exe), *args], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    return run


def _dh(L, d, V):
    """The dh contraction of Eq. 10 in one chunk (V columns)."""
    regions = min(32 * -(-L // 256) * -(-d // 256), 320)
    return (L, d, -(-V // 256) * 256, 0, regions, 1, 1)


def _forward(L, din, dout, r):
    return (L, dout, din, r, 160, 0, 1)


def _input_grad(L, din, dout, r):
    return (L, din, dout, r, 160, 1, 0)


# the shapes of the GPU tests (test_gpu_ce.py, test_gpu_lora_proj.py)
GROUPED_PIECES = [_dh(4200, 512, 32000), _dh(4097, 512, 20000), _dh(4352, 520, 20000), _dh(6000, 384, 50257),
                  _forward(4352, 14336, 512, 16), _input_grad(4352, 512, 14336, 16), _forward(4737, 6784, 320, 16)]


def test_pieces_of_grouped_tiles_are_where_the_sum_reads_them(walk):
    """Shapes that run in K pieces, in row groups and more than one column tile
    wide: there the order of the tiles is not the order of the regions."""
    for shape, (pieces, group, tiles_n, bad) in zip(GROUPED_PIECES, walk(GROUPED_PIECES)):
        assert pieces > 1 and group > 0 and tiles_n > 1, shape
        assert bad == 0, shape


def test_pieces_over_a_grid_of_shapes(walk):
    shapes = []
    for L in (1, 33, 128, 129, 257, 1000, 2049, 4097, 4200, 5000, 6144, 8191, 12000):
        for d in (8, 64, 200, 264, 384, 512, 520, 640, 736, 1032, 3584, 5120):
            shapes += [_dh(L, d, V) for V in (600, 8192, 20011, 50257, 152064)]
            shapes += [f(L, a, b, 16) for f in (_forward, _input_grad) for a, b in ((d, 8192), (14336, d), (d, d))]
    got = walk(shapes)
    assert len(got) == len(shapes)
    for shape, (_, _, _, bad) in zip(shapes, got):
        assert bad == 0, shape
    assert sum(p > 1 and g > 0 and n > 1 for p, g, n, _ in got) >= 20


def test_eq10_chains_and_pairs_stay_within_their_bounds(walk):
    """Whatever the plan: chunks no wider than the workspace is laid out for,
    no accumulation of dh over more than 65,536 columns, and no more (max, sum)
    pairs than there is room for; also on parts with fewer or more SMs."""
    shapes = [(L, d, V, min(32 * -(-L // 256) * -(-d // 256), 320), sms)
              for L in (1, 40, 93, 129, 300, 403, 600, 1024, 1500, 2048, 4097, 5888, 8192, 32768)
              for d in (8, 512, 1032, 1544, 3584, 5120, 8192) for V in (1, 300, 8192, 66000, 152064, 262144, 1000000)
              for sms in (148, 152, 160, 72)]
    got = walk(shapes, "eq10")
    assert len(got) == len(shapes)
    for shape, (vc, vmax, chain, pairs, room) in zip(shapes, got):
        assert 0 < vc <= vmax and chain <= 65536 and pairs <= room, shape
    assert walk([(403, 3584, 152064, 320, 152)], "eq10")[0][0] == 152064  # in pieces: one chunk
    assert walk([(2048, 3584, 152064, 320, 152)], "eq10")[0][0] == 50688  # whole tiles: three
