"""The height of the decode tiles, and the border between the 64-token tiles and the CTA pairs on matrices with a long K, evaluated
on the host with the capacities of a B200.  Lower tiles only where K is long enough for their even load to show; the pairs serve what
they were measured to be faster on, and the sizes at which they would leave much of the chip idle, or take a whole round for a few
tiles, stay with the tiles."""
import pytest

from tests.helpers import host_program

PROGRAM = r"""
#include "pair_plan.h"
#include "tile_plan.h"
#include <cstdio>
int main() {
    const int pair_capacity[] = {0, 74, 33, 22, 15}, tile_capacity[] = {0, 296, 296, 270, 296, 260, 270, 210, 264};
    long long M, N, K; int full;
    while (scanf("%d %lld %lld %lld", &full, &M, &N, &K) == 4) {
        if (M <= 32) {
            printf("%d\n", dps::tile_plan::low_rows(full, N, K, M <= 16 ? 16 : 32, 148));
            continue;
        }
        const auto p = dps::pair_plan::make_plan(full, M, N, K, pair_capacity);
        const long long pair_tiles = (N + 255) / 256 * ((M + p.tokens - 1) / p.tokens), tiles = (N + 127) / 128;
        const int kb = full ? 64 : 128, split = dps::tile_plan::choose_split(tiles, (int)((K + kb - 1) / kb), tile_capacity, full ? 5 : 4);
        const auto pairs = dps::tile_plan::turns(pair_tiles, p.split, pair_capacity[1]);
        const auto alone = dps::tile_plan::turns(tiles, split, tile_capacity[1]);
        printf("%d\n", (int)dps::tile_plan::pairs_for_long_k(pairs, alone));
    }
}
"""
# 256-row tiles: where the pairs are the faster ones
FASTER = [*range(20, 23), *range(27, 34), *range(46, 75), *range(149, 223), *range(297, 371)]


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("plan"), PROGRAM)
    return lambda cases: [answer for (answer,) in run(cases)]


@pytest.mark.parametrize("K", [16384, 17920, 28672, 53248])
def test_pairs_serve_a_long_k_where_they_fill_the_chip(ask, K):
    for full in (0, 1):
        for M in (33, 48, 64):
            tiles = range(20, 371)
            got = ask([(full, M, 256 * t, K) for t in tiles] + [(full, M, 256 * t - 248, K) for t in tiles])   # (8 rows in the last tile)
            assert [t for t, g in zip(tiles, got) if g] == FASTER
            short = [t for t, g in zip(tiles, got[len(tiles):]) if g]
            assert set(short) <= set(FASTER) and set(range(28, 33)) | set(range(48, 73)) <= set(short)


def test_sizes_that_lost(ask):
    lost = [(f, 64, n, k) for f in (0, 1) for n in (8456, 10240, 11264, 19200, 20480, 28672) for k in (16384, 28672)]
    assert not any(ask(lost))


def test_tile_heights(ask):
    # (mode, tokens, rows, K): the height; a short K keeps 128 rows whatever the rows
    for case, rows in [((1, 12, 22016, 4096), 88), ((1, 32, 22016, 4096), 88), ((1, 12, 57344, 8192), 104), ((1, 32, 57344, 8192), 128), ((0, 12, 57344, 8192), 104),
                       ((0, 32, 57344, 8192), 128), ((0, 12, 22016, 4096), 128), ((1, 12, 18944, 4096), 128), ((1, 12, 18952, 4096), 88), ((1, 24, 38016, 1536), 88)]:
        assert ask([case]) == [rows], case
    short = [(f, M, N, K) for f in (0, 1) for M in (12, 24) for N in range(18952, 130000, 1000) for K in (16, 256, 768, 1024, 1520)]
    assert set(ask(short)) == {128}
    tall = ask([(f, M, N, 4096) for f in (0, 1) for M in (12, 24) for N in range(18952, 300000, 504)])
    assert all(r % 8 == 0 and 88 <= r <= 128 for r in tall) and len(set(tall)) > 4
