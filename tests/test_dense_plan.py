"""The division of the prompt pass's dense products over pairs of CTAs (host arithmetic, no GPU): every (tile, chunk) is
multiplied once, every pair waits only for what pairs with a lower number compute first, and the order in which a tile's
chunks are added does not depend on the number of positions."""

import random

import numpy as np
import pytest

from paper_2506_03700_b200 import binding

WIDE, PAIRED = 256, 128   # weight rows of a tile; where gate and up rows share one
SHAPES = [  # (N, per tile, K): QKV, O, gate / up and down of the 8B, 1B and 13B shapes, and odd ones
    (6144, WIDE, 4096), (4096, WIDE, 4096), (14336, PAIRED, 4096), (4096, WIDE, 14336),
    (3072, WIDE, 2048), (2048, WIDE, 2048), (8192, PAIRED, 2048), (2048, WIDE, 8192),
    (15360, WIDE, 5120), (5120, WIDE, 5120), (13824, PAIRED, 5120), (5120, WIDE, 13824),
    (256, WIDE, 704), (64, PAIRED, 64), (1000, WIDE, 3008), (9472, PAIRED, 1088), (18944, WIDE, 1600),
]
ROWS = [1, 9, 31, 33, 64, 96, 200, 256, 257, 300, 512, 513, 777, 800, 1024, 1025, 1280, 1500, 1792, 2000, 2047, 2048]


def group_begin(plan, i):
    return i * plan["chunks"] // plan["groups"]


def run(rows, N, per_tile, K, pairs):
    """Multiplies and adds as the kernel does, with one float32 number for the product of every chunk; returns the plan and
    the sum of every tile.  Fails where something is multiplied twice, missing, or not yet there when it is needed."""
    plan, _ = binding.debug_dense_plan(rows, N, per_tile, K, pairs, 0)
    value = np.random.default_rng(K).normal(size=plan["chunks"]).astype(np.float32)
    begins = [group_begin(plan, i) for i in range(plan["groups"] + 1)]
    published, sums, done = {}, {}, set()     # pair -> (tile, end, total, group so far); tile -> sum; (tile, chunk)
    for pair in range(plan["pairs"]):
        segs = binding.debug_dense_plan(rows, N, per_tile, K, pairs, pair)[1]
        assert [i for i, (_, _, c1) in enumerate(segs) if c1 < plan["chunks"]] in ([], [0])   # published once, and first
        for tile, c0, c1 in segs:
            total, acc, first_pair = None, np.float32(0), pair
            if c0 > 0:                        # the pieces before this one: lower pairs, in an unbroken row from chunk 0
                need = c0
                while need > 0:
                    first_pair -= 1
                    t, end, _, _, start = published[first_pair]
                    assert t == tile and end == need
                    need = start
            g = max(i for i, b in enumerate(begins[:-1]) if b <= c0)
            middle = c0 > 0 and c1 < plan["chunks"]
            if middle:
                assert begins[g] == c0 and begins[g + 1] == c1
            if c0 > begins[g]:
                assert first_pair == pair - 1 and published[pair - 1][4] == 0
                acc = published[pair - 1][3]
            if c0 > 0 and not middle and g > 0:
                for p in range(first_pair, pair):
                    total = published[p][2] if total is None else np.float32(total + published[p][2])
                assert pair - first_pair <= 3
            for c in range(c0, c1):
                assert (tile, c) not in done
                done.add((tile, c))
                acc = np.float32(acc + value[c])
                if c + 1 == begins[g + 1]:
                    total = acc if total is None else np.float32(total + acc)
                    acc, g = np.float32(0), g + 1
            if c1 == plan["chunks"]:
                sums[tile] = total
            else:
                assert pair not in published
                published[pair] = (tile, c1, total, acc, c0)
    assert len(done) == plan["tiles"] * plan["chunks"] and len(sums) == plan["tiles"]
    return plan, sums


def check(rows, N, per_tile, K, pairs):
    plan, sums = run(rows, N, per_tile, K, pairs)
    assert 32 <= plan["nt"] <= 256 and plan["nt"] % 32 == 0 and plan["nt"] * plan["mt"] >= rows
    assert plan["tiles"] == plan["mt"] * -(-N // per_tile) and 1 <= plan["pairs"] <= pairs
    assert len(set(sums.values())) == 1
    assert plan["ck"] == min(8, max(4, K // 512)) and plan["chunks"] == -(-(K // 64) // plan["ck"])
    return plan["groups"], sums[0]


@pytest.mark.parametrize("N,per_tile,K", SHAPES)
@pytest.mark.parametrize("pairs", [74, 66, 13, 1])
def test_every_chunk_once_and_the_same_order_for_every_number_of_positions(N, per_tile, K, pairs):
    assert len({check(rows, N, per_tile, K, pairs) for rows in (ROWS if pairs == 74 else ROWS[::3])}) == 1


def test_random_shapes():
    rng = random.Random(7)
    for _ in range(150):
        N, per_tile, K = rng.randint(1, 400) * 64, rng.choice([WIDE, PAIRED]), rng.randint(1, 230) * 64
        pairs = rng.choice([74, 74, rng.randint(1, 76)])
        assert len({check(rng.randint(1, 2048), N, per_tile, K, pairs) for _ in range(4)}) == 1


def test_bad_arguments():
    for args in ((0, 256, 256, 256, 74, 0), (2049, 256, 256, 256, 74, 0), (64, 256, 100, 256, 74, 0), (64, 256, 256, 100, 74, 0), (64, 256, 256, 256, 74, 74)):
        with pytest.raises(binding.AdaError) as e:
            binding.debug_dense_plan(*args)
        assert e.value.code == -1
