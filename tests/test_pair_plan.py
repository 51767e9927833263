"""The tile plan of the CTA-pair linear, evaluated on the host over its whole range of sizes: every width is one that the
instruction has, the rings fit shared memory, and the tiles and pieces cover every token exactly once."""
import random

import pytest

from tests.helpers import host_program

PROGRAM = r"""
#include "pair_plan.h"
#include <cstdio>
using namespace dps::pair_plan;
int main() {
    long long M, N, K, A; int full, E;
    int cap[kMaxSplit + 1];
    char kind;
    while (scanf(" %c", &kind) == 1) {
        if (kind == 'd') {
            if (scanf("%d %lld %lld %lld %d %d %d %d", &full, &M, &N, &K, cap + 1, cap + 2, cap + 3, cap + 4) != 8) return 1;
            const Plan p = make_plan(full, M, N, K, cap);
            const Rings r = size_rings(full, p.tokens);
            printf("%d %d %d %d %d %d\n", p.tokens, p.tail_parts, p.tail_tokens, p.split, r.units, r.x_slots);
        } else {
            if (scanf("%d %lld %lld %d", &full, &A, &N, &E) != 4) return 1;
            const int t = grouped_width(full, A, N, E, 74);
            const Rings f = size_rings(false, t), g = size_rings(true, t);
            printf("%d %d %d %d %d\n", t, f.units, f.x_slots, g.units, g.x_slots);
        }
    }
}
"""
# resident clusters of 1 .. 4 pairs: a whole device, one with few clusters, a small one without any larger cluster
CAPACITIES = [(0, 74, 33, 16, 16), (0, 66, 30, 14, 14), (0, 9, 4, 2, 2), (0, 3, 0, 0, 0)]


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    return host_program(tmp_path_factory.mktemp("plan"), PROGRAM)


def check_rings(full, tokens, units, x_slots):
    unit = 128 * 128 * (2 if full else 1)
    assert units >= 2 and units % 2 == 0 and units <= 12 and (4 if tokens <= 256 else 3) <= x_slots <= 8
    assert units * unit + x_slots * tokens * 128 + 4 * 32 * 64 + 1024 <= 222 * 1024


def check_dense(full, M, N, K, cap, answer):
    tokens, parts, tail_tokens, split, units, x_slots = answer
    assert tokens % 32 == 0 and tail_tokens % 32 == 0 and 32 <= tail_tokens <= tokens
    # wide tiles: two MMAs each, which a piece must do with one of; K is not split
    assert 32 <= tokens <= 256 or (tokens in (320, 384) and M > 256 and split == 1 and (parts == 1 or tail_tokens <= tokens // 2))
    check_rings(full, tokens, units, x_slots)
    row_tiles, tok_tiles = -(-N // 256), -(-M // tokens)
    tiles, pairs = row_tiles * tok_tiles, cap[1]
    assert 1 <= split <= 4 and (split == 1 or (tiles <= cap[split] and -(-K // 128) >= 2 * split and parts == 1))
    if parts > 1:
        tail = tiles % pairs
        assert tail and tail * parts <= pairs and parts * tail_tokens >= tokens
    # every token of a token tile in exactly one piece
    for first in {0, (tok_tiles - 1) * tokens}:
        end = min(M, first + tokens)
        covered = sum(max(0, min(tail_tokens, end - first - i * tail_tokens)) for i in range(parts))
        assert covered == end - first


def test_dense_plans_over_the_range(plan):
    rng = random.Random(5)
    cases = []
    for _ in range(4000):
        M = int(2 ** rng.uniform(0, 14))
        N = 8 * int(2 ** rng.uniform(0, 14))
        K = 16 * int(2 ** rng.uniform(0, 11))
        cases.append((rng.randrange(2), M, N, K, rng.choice(CAPACITIES)))
    cases += [(f, M, N, 4096, CAPACITIES[0]) for f in (0, 1) for M in range(1, 700) for N in (4096, 18944)]
    cases += [(f, M, N, 4096, c) for f in (0, 1) for M in (257, 320, 384, 700, 1100, 1536, 2999, 8192) for N in range(256, 24000, 744) for c in CAPACITIES]
    answers = plan([f"d {f} {M} {N} {K} {c[1]} {c[2]} {c[3]} {c[4]}" for f, M, N, K, c in cases])
    assert len(answers) == len(cases)
    for case, answer in zip(cases, answers):
        check_dense(*case, answer)
    assert any(a[1] > 1 for a in answers) and any(a[3] > 1 for a in answers)
    # wide tiles, whole and in pieces, with every number of pairs
    assert {(c[4], a[1] > 1) for c, a in zip(cases, answers) if a[0] > 256} == {(c, cut) for c in CAPACITIES for cut in (False, True)}


@pytest.mark.parametrize("tokens", ["16", "48", "112", "256", "300", "384"])
def test_forced_widths_are_widths_there_are(plan, tokens):
    for M, answer in zip((500, 31), plan(["d 0 500 4096 4096 74 33 16 16", "d 1 31 512 2064 74 33 16 16"], DPS_PAIR_TOKENS=tokens), strict=True):
        assert answer[0] % 32 == 0 and (32 <= answer[0] <= 256 or (M > 256 and answer[0] == max(320, int(tokens)))) and answer[2] % 32 == 0


def test_grouped_widths(plan):
    cases = [(f, A, N, E) for f in (0, 1) for N in (8, 4096, 40000) for E in (1, 3, 8, 64, 1024)
             for A in sorted({1, 47 * E, 48 * E, 49 * E, 100 * E + 7, 200 * E, 256 * E, 257 * E, 5000 * E})]
    for (f, A, N, E), (tokens, *rings) in zip(cases, plan([f"g {f} {A} {N} {E}" for f, A, N, E in cases]), strict=True):
        assert tokens % 32 == 0 and 32 <= tokens <= 256, (A, E)
        check_rings(False, tokens, *rings[:2])
        check_rings(True, tokens, *rings[2:])


def test_an_uneven_routing_does_not_add_a_round(plan):
    """Few rows per expert: an expert with a good part of all rows still has one token tile, so that the one round that the border counted stays one; wider tiles only below 48 rows."""
    for full, E, N, rows, share in ((0, 4, 4096, 40, 0.47), (1, 4, 4096, 40, 0.47), (1, 8, 2304, 40, 0.38), (0, 16, 1024, 40, 0.15), (1, 3, 15496, 40, 0.53), (1, 64, 256, 47, 0.04)):
        assert plan([f"g {full} {rows * E} {N} {E}"])[0][0] >= share * rows * E, (full, E, N, rows)
    assert [plan([f"g {f} {rows * 8} {N} 8"])[0][0] for f, rows, N in ((0, 24, 14336), (1, 24, 14336), (0, 24, 2304), (1, 24, 2304), (0, 48, 2304), (1, 48, 2304))] == [64, 96, 96, 128, 96, 96]
