"""The tile plan of the CTA-pair linear, evaluated on the host over its whole range of sizes: every width is one that the
instruction has, the rings fit shared memory, and the tiles and pieces cover every token exactly once."""
import random
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parents[1] / "paper_2609_34380_b200" / "csrc"
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
            if (scanf("%lld %d", &A, &E) != 2) return 1;
            const int t = grouped_tokens(A, E);
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
    gxx = shutil.which("g++")
    assert gxx
    where = tmp_path_factory.mktemp("plan")
    (where / "plan.cpp").write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", str(CSRC), str(where / "plan.cpp"), "-o", str(where / "plan")], check=True)

    def ask(lines, **env):
        out = subprocess.run([str(where / "plan")], input="\n".join(lines), text=True, capture_output=True, check=True, env=env)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return ask


def check_rings(full, tokens, units, x_slots):
    unit = 128 * 128 * (2 if full else 1)
    assert units >= 2 and units % 2 == 0 and units <= 12 and 4 <= x_slots <= 8
    assert units * unit + x_slots * tokens * 128 + 4 * 32 * 64 + 1024 <= 222 * 1024


def check_dense(full, M, N, K, cap, answer):
    tokens, parts, tail_tokens, split, units, x_slots = answer
    assert tokens % 32 == 0 and 32 <= tokens <= 256 and tail_tokens % 32 == 0 and 32 <= tail_tokens <= tokens
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
    answers = plan([f"d {f} {M} {N} {K} {c[1]} {c[2]} {c[3]} {c[4]}" for f, M, N, K, c in cases])
    assert len(answers) == len(cases)
    for case, answer in zip(cases, answers):
        check_dense(*case, answer)
    assert any(a[1] > 1 for a in answers) and any(a[3] > 1 for a in answers)


@pytest.mark.parametrize("tokens", ["16", "48", "112", "256", "300"])
def test_forced_widths_are_widths_there_are(plan, tokens):
    for answer in plan(["d 0 500 4096 4096 74 33 16 16", "d 1 31 512 2064 74 33 16 16"], DPS_PAIR_TOKENS=tokens):
        assert answer[0] % 32 == 0 and 32 <= answer[0] <= 256 and answer[2] % 32 == 0


def test_grouped_widths(plan):
    cases = [(A, E) for E in (1, 3, 8, 64, 1024) for A in sorted({1, 47 * E, 48 * E, 49 * E, 100 * E + 7, 200 * E, 256 * E, 257 * E, 5000 * E})]
    for (A, E), (tokens, *rings) in zip(cases, plan([f"g {A} {E}" for A, E in cases])):
        assert tokens % 32 == 0 and 32 <= tokens <= 256, (A, E)
        check_rings(False, tokens, *rings[:2])
        check_rings(True, tokens, *rings[2:])
