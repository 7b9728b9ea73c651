"""The rule that picks tiles and parts of a dense product (no GPU needed): every tile of its table is the choice for some
product, has a tensor map of its height, and parts of the reduction dimension stay long enough."""
import os
import random
import re

from helpers import gemm_plan

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_01028_b200", "csrc", "gemm_plan.h")


def _table():
    return {(int(a), int(b)) for a, b in re.findall(r"consider\((\d+), (\d), \d+\);", open(HEADER).read())}


def test_every_tile_of_the_table_is_chosen_by_some_product():
    rng = random.Random(1)
    chosen = {gemm_plan(rng.randint(1, 2048), rng.randint(32, 22016), 8 * rng.randint(8, 1376))[:2] for _ in range(4000)}
    assert chosen == _table() and len(chosen) == 9


def test_plans_cover_the_product():
    boxes = {int(b) for b in re.search(r"kWBoxRows\[\] = \{([^}]*)\}", open(HEADER).read()).group(1).split(",")}
    assert boxes == {bn // cg for bn, cg in _table()}  # one tensor map for each height, and none for another
    rng = random.Random(2)
    for _ in range(2000):
        M, N, K, most = rng.randint(1, 2048), rng.randint(1, 22016), 8 * rng.randint(1, 1376), rng.randint(1, 8)
        p = gemm_plan(M, N, K, most, sms=rng.choice([2, 132, 148, 160]))
        assert p.bn // p.cg in boxes and p.bn % 32 == 0
        assert p.m_tiles == -(-M // (128 * p.cg)) and p.tiles == p.m_tiles * -(-N // p.bn)
        assert 1 <= p.parts <= most and (p.parts == 1 or -(-K // 64) // p.parts >= 8)
