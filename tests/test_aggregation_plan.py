"""The aggregation's tiles and the bytes its blocks copy stay inside the packed rows (compiled from the header that the
kernels use; no GPU needed)."""
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cinttypes>
#include <cstdio>
#include "tq_aggregation_plan.h"
int main() {
    int bits, n, apply;
    uint64_t d;
    while (std::scanf("%d %" SCNu64 " %d %d", &bits, &d, &n, &apply) == 4) {
        const tq::AggregationPlan p = tq::plan_aggregation(bits, d, n, apply);
        const uint64_t row = ((d * bits + 31) / 32 + 3) / 4 * 16, tile = tq::tile_bytes(bits, p.units), last = (p.blocks - 1) * tile;
        std::printf("%d %d %" PRIu64 " %d %" PRIu64 " %" PRIu64 " %u\n", p.bulk, p.units, p.blocks, tq::unit_elems(bits), row, last,
                    last < row ? tq::tile_bytes_in_row(row, last, tile) : 0u);
    }
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    where = tmp_path_factory.mktemp("plan")
    (where / "plan.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", "-I", os.path.join(ROOT, "paper_2402_01798_b200", "csrc"), str(where / "plan.cpp"),
                    "-o", str(where / "plan")], check=True)

    def ask(calls):
        out = subprocess.run([str(where / "plan")], input="".join("%d %d %d %d\n" % c for c in calls), capture_output=True, text=True, check=True)
        return [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    return ask


def test_every_tile_starts_inside_the_row(plan):
    """d just above a multiple of the largest tile, where the smaller tiles of the fused update used to start beyond the row:
    25 600 001 x 16, 4 bits, ended 2032 bytes behind it."""
    r = random.Random(5)
    sizes = [k * 4096 + o for k in (1, 295, 296, 300, 1365, 4095, 4096, 4097, 6250)
             for o in (-1, 0, 1, 5, 31, 33, 511, 513, 1023, 1024, 1025, 2047, 2048, 2049, 3071, 3073)]
    sizes += [1, 7, 5_592_384, 11_200_001, 25_600_001, 2 ** 40] + [int(2 ** r.uniform(0, 33)) for _ in range(300)]
    calls = [(bits, d, n, apply) for bits in (1, 2, 3, 4) for d in sizes for n in (1, 32, 33, 64) for apply in (0, 1)]
    forms = set()
    for (bits, d, n, apply), (bulk, units, blocks, elems, row, last, copied) in zip(calls, plan(calls), strict=True):
        per_block = 128 * units * elems
        assert (blocks - 1) * per_block < d <= blocks * per_block, (bits, d, n, apply)       # each block has an element, all have one
        assert last < row and 0 < copied <= 128 * units * (3 if bits == 3 else 4) and last + copied == row
        assert copied % 16 == 0 and last % 16 == 0                                           # as a bulk copy needs
        forms.add((bits, bulk, units))
    assert {(4, 1, 1), (4, 1, 2), (4, 1, 4), (2, 1, 1), (2, 1, 2), (4, 0, 1), (1, 1, 1)} <= forms
