"""Which rows of a matrix the CTA pairs take at 17 to 128 tokens (pair_plan.h): the rule's edges, and that a cut leaves whole tiles on one side."""
import random

import pytest

from tests.helpers import host_program

PROGRAM = r"""
#include "pair_plan.h"
#include <cstdio>
int main(int argc, char**) {
    long long M, N, K; int full, pairs;
    int E;
    while (argc > 1 && scanf("%d %lld %lld %lld %d %d", &full, &M, &N, &K, &E, &pairs) == 6)      // (M rows over E experts)
        printf("%d 0\n", (int)dps::pair_plan::grouped_on_pairs(full, M, N, K, E, pairs));
    while (scanf("%d %lld %lld %lld %d", &full, &M, &N, &K, &pairs) == 5) {
        const auto s = dps::pair_plan::share_rows(full, M, N, K, pairs);
        printf("%d %lld %d\n", (int)s.pairs, (long long)s.rows, (int)dps::pair_plan::may_share_rows(M, N, 2 * pairs));
    }
}
"""
ROUND = 74 * 256
# (full, M, N, K): None: the other rules decide; 0: pairs, one launch; n: pairs up to there, the rest by itself
EDGES = {(1, 64, ROUND - 256, 8192): 0, (0, 33, 60 * 256, 3072): 0, (0, 33, 59 * 256, 3072): None, (1, 64, 60 * 256, 3056): None, (1, 32, 60 * 256, 8192): None,
         (1, 65, 60 * 256, 8192): None, (0, 64, 60 * 256, 16384): None, (1, 64, ROUND, 8192): 0, (1, 64, ROUND + 8, 8192): ROUND, (1, 33, 86 * 256, 2048): None, (1, 33, 86 * 256, 4096): None,
         (1, 64, 86 * 256, 5120): ROUND, (1, 64, 112 * 256, 5120): 0, (1, 64, 224 * 256, 8192): 3 * ROUND, (1, 64, 75 * 256, 16384): None,
         (1, 16, 224 * 256, 8192): None, (1, 17, 224 * 256, 8192): 3 * ROUND, (1, 17, 224 * 256, 1536): None, (1, 32, 226 * 256, 4096): None, (1, 32, 158 * 256, 4096): 2 * ROUND, (1, 33, 158 * 256, 2048): 0, (0, 33, 158 * 256, 2048): None, (1, 32, 86 * 256, 4096): None,
         (1, 32, 86 * 256, 8192): ROUND, (0, 64, 86 * 256, 4096): None, (0, 64, 76 * 256, 8192): ROUND, (0, 64, 150 * 256, 4096): 0, (0, 64, 224 * 256, 8192): None, (0, 64, 296 * 256, 8192): None,
         (0, 32, 224 * 256, 8192): None, (1, 96, 76 * 256, 4096): ROUND, (1, 96, 86 * 256, 4096): None, (0, 128, 224 * 256, 8192): 3 * ROUND,
         (1, 129, 224 * 256, 8192): None}


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    run = host_program(tmp_path_factory.mktemp("rows"), PROGRAM)
    return lambda cases, *argv, whole=False, **env: [answer[:None if whole else 2] for answer in run(cases, *argv, **env)]


def test_edges(ask):
    for (case, want), (pairs, rows) in zip(EDGES.items(), ask([(*c, 74) for c in EDGES])):
        assert (None if not pairs else rows) == want, case


def test_a_cut_is_whole_rounds_and_a_rest(ask):
    rng = random.Random(4)
    cases = [(rng.randrange(2), int(2 ** rng.uniform(0, 10)), 8 * int(2 ** rng.uniform(0, 14.5)), 16 * int(2 ** rng.uniform(0, 11)), rng.choice((74, 66, 9))) for _ in range(4000)]
    for env in ({}, {"DPS_ROW_CUT": "1"}):
        cuts = 0
        for (full, M, N, K, pairs), (taken, rows) in zip(cases, ask(cases, **env)):
            assert not rows or (taken and 0 < rows < N and rows % (256 * pairs) == 0 and N - rows < 256 * pairs and 16 < M <= 256)
            cuts += rows > 0
        assert cuts > 20
    assert all(answer == (0, 0) for answer in ask(cases, DPS_ROW_CUT="0"))


def test_grouped_launches_on_pairs(ask):
    # (full, rows, N, K, experts)
    edges = {(0, 48 * 8, 4096, 64, 8): 1, (0, 47 * 8, 4096, 14336, 8): 0, (0, 20 * 8, 28672, 4096, 8): 1, (0, 20 * 8 - 1, 28672, 4096, 8): 0,
             (1, 12 * 8, 28672, 4096, 8): 1, (1, 12 * 8 - 1, 28672, 4096, 8): 0, (1, 30 * 8, 4096, 14336, 8): 0, (0, 30 * 4, 4096, 8192, 4): 1,
             (0, 30 * 4, 4096, 3056, 4): 0, (0, 30 * 8, 264, 8192, 8): 0, (0, 30 * 64, 2816, 2048, 64): 1, (1, 30 * 8, 2816, 8192, 8): 0, (1, 30 * 4, 16384, 4096, 4): 0}
    assert [pairs for pairs, _ in ask([(*c, 74) for c in edges], "grouped")] == list(edges.values())


def test_grouped_launches_count_the_turns_of_either_kernel(ask):
    """Below eight rounds no shape goes to the pairs that the tiles of 128 rows serve in as many turns or fewer, each counted as its kernel cuts the rows."""
    cases = [(full, 30 * E, N, K, E) for full in (0, 1) for E in (4, 8, 12, 16, 32, 64, 100, 256) for N in [*range(8, 512, 56), *range(512, 8193, 32)] for K in (1024, 8192)]
    given = 0
    for (full, A, N, K, E), (pairs, _) in zip(cases, ask([(*c, 74) for c in cases], "grouped"), strict=True):
        rounds, turns = -(-E * -(-N // 256) // 74), 2 * -(-E * -(-N // 128) // (4 * 74))
        assert rounds == 1 or rounds >= 8 or pairs == (rounds < turns), (full, A, N, K, E)
        given += pairs
    assert given > len(cases) // 4
    # three rounds against a wave; seven against three; the same with a shape that fills its tiles; eleven against five waves
    edges = {(0, 24 * 32, 1152, 2048, 32): 0, (1, 13 * 8, 4736, 4096, 8): 0, (1, 24 * 16, 6976, 1024, 16): 0, (1, 24 * 16, 7168, 1024, 16): 1, (0, 24 * 64, 2880, 2048, 64): 1}
    assert [pairs for pairs, _ in ask([(*c, 74) for c in edges], "grouped")] == list(edges.values())


def test_grouped_launches_with_a_long_routing_stay_on_the_tiles(ask):
    edges = {(0, 24 * 256, 1152, 1024, 256): 1, (0, 24 * 257, 1152, 1024, 257): 0, (1, 13 * 512, 384, 1024, 512): 0, (0, 47 * 1024, 128, 1024, 1024): 0, (0, 48 * 512, 384, 1024, 512): 1}
    assert [pairs for pairs, _ in ask([(*c, 74) for c in edges], "grouped")] == list(edges.values())


def test_a_rest_is_cut_off_only_where_that_was_measured_to_pay(ask):
    """As measured (the table beside the rule): the rests that a launch of their own makes slower stay, those that gain 2 us and more are cut off."""
    pays = [(0, 64, 2, 4, 8192), (0, 64, 2, 4, 14336), (0, 64, 2, 11, 8192), (0, 64, 2, 20, 8192), (0, 64, 2, 20, 14336), (0, 64, 2, 30, 14336), (1, 64, 1, 4, 8192), (1, 64, 1, 16, 8192), (1, 64, 1, 26, 8192), (1, 64, 1, 26, 14336),
            (1, 64, 2, 16, 14336), (1, 24, 2, 10, 8192), (1, 24, 2, 30, 8192), (1, 24, 2, 30, 14336)]
    loses = [(0, 64, 2, r, K) for r in (40, 50, 60, 73) for K in (4096, 8192, 14336)] + [(0, 64, 2, r, 4096) for r in (4, 11, 20, 30)]
    loses += [(1, 64, n, r, K) for n in (1, 2) for r in (35, 45, 51) for K in (8192, 14336)] + [(1, 24, 2, 45, K) for K in (8192, 14336)]
    for cases, cut in ((pays, True), (loses, False)):
        for (full, M, rounds, rest, K), (pairs, rows) in zip(cases, ask([(f, M, (74 * n + r) * 256 - 96, K, 74) for f, M, n, r, K in cases])):
            assert pairs and (rows > 0) == cut, (full, M, rounds, rest, K)
    # anywhere else: never most of a round, and with as many K steps never a longer rest where a shorter one stays
    for full in (0, 1):
        for M in (17, 32, 33, 64):
            for n in (1, 2, 5):
                for K in (2048, 4096, 8192, 12288, 16368):
                    rows = [r for taken, r in ask([(full, M, (74 * n + rest) * 256, K, 74) for rest in range(1, 74)]) if taken]
                    longest = sum(r > 0 for r in rows)
                    assert all(r > 0 for r in rows[:longest]) and longest <= 37, (full, M, n, K, longest)


def test_a_tile_for_every_pair_is_one_round(ask):
    """74 row tiles, every pair busy: the rule of 60 to 73, not that of a round and a rest."""
    for full in (0, 1):
        for M in (33, 64):
            for N in (ROUND - 248, ROUND - 96, ROUND):
                cases = [(full, M, N, K, 74) for K in (3056, 3072, 4096, 5104, 8192, 14336)]
                assert ask(cases) == [(0, 0)] + [(1, 0)] * 5, (full, M, N)
    assert ask([(f, M, ROUND, K, 74) for f in (0, 1) for M in (17, 32, 65, 128) for K in (4096, 8192)]) == [(0, 0)] * 16


def test_calls_that_cannot_share_do_not_ask(ask):
    cases = [(full, M, N, K, 74) for full in (0, 1) for M in (8, 16, 17, 33, 64, 65, 128, 129, 200, 256, 257) for N in (4096, 9464, 9472, 15112, 18944, 22016, 57344) for K in (2048, 8192, 16384)]
    for env, most in (({}, 128), ({"DPS_ROW_CUT": "1"}, 256)):
        for (full, M, N, K, _), (pairs, rows, asked) in zip(cases, ask(cases, whole=True, **env), strict=True):
            assert asked == (16 < M <= most and N >= 9472) and (asked or not pairs), (full, M, N, K)
