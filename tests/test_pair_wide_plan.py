"""The CTA pairs' plan with wide tiles: the widths that exist, rings that fit, accumulators and A ring within tensor memory, pieces that fit a half."""
import random

from tests.helpers import host_program

PROGRAM = r"""
#include "pair_plan.h"
#include <cstdio>
using namespace dps::pair_plan;
int main() {
    long long M, N, K; int full;
    const int cap[kMaxSplit + 1] = {0, 74, 33, 16, 16};
    while (scanf("%d %lld %lld %lld", &full, &M, &N, &K) == 4) {
        const Plan p = make_plan(full, M, N, K, cap);
        const Rings r = size_rings(full, p.tokens);
        printf("%d %d %d %d %d %d %d %d\n", p.tokens, mma_tokens(p.tokens), p.tokens > kMaxTokens ? kWideASteps : kASteps, p.tail_parts, p.tail_tokens, p.split, r.units, r.x_slots);
    }
}
"""


def test_wide_plans_over_the_range(tmp_path):
    run = host_program(tmp_path, PROGRAM)
    rng = random.Random(3)
    cases = [(rng.randrange(2), int(2 ** rng.uniform(0, 14)), 8 * int(2 ** rng.uniform(0, 13)), 16 * int(2 ** rng.uniform(0, 11))) for _ in range(3000)]
    cases += [(f, M, 12288, 4096) for f in (0, 1) for M in (1, 64, 256, 257, 320, 321, 384, 385, 640, 8192)]
    wide = 0
    for (full, M, N, K), (tokens, mma, a, parts, tail, split, units, slots) in zip(cases, run(cases), strict=True):
        assert 32 <= mma <= 256 and mma % 32 == 0 and tokens in (mma, 2 * mma)
        assert tokens <= 256 or (tokens in (320, 384) and M > 256 and split == 1)
        assert tokens + 64 * a <= 512 and a == (2 if tokens > 256 else 4)
        assert units >= 2 and units % 2 == 0 and slots >= (3 if tokens > 256 else 4)
        assert units * 128 * 128 * (1 + full) + slots * tokens * 128 + 4 * 32 * 64 + 1024 <= 222 * 1024
        assert parts == 1 or (tail <= mma and parts * tail >= tokens)
        wide += tokens > 256
    assert wide
