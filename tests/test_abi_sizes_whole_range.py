"""The stream bound over the whole block range equals the sum over its parts."""
import random

import torch

from paper_2601_20113_gb300 import dls


def _align(x):
    return -(-x // 16) * 16


def test_bound_of_the_whole_range_is_the_sum_of_its_parts():
    r = random.Random(1)
    seen = 0
    while seen < 100:
        d = [r.randint(1, 40) for _ in range(4)]
        b = [r.randint(1, min(x, 8)) for x in d]
        nv = r.randint(1, 3)
        nb = nv
        for x, y in zip(d, b):
            nb *= -(-x // y)
        if min(b[0] * b[1] * b[2], b[3]) > 32 or nb < 2:
            continue
        seen += 1
        p = dls.make_params((nv, d[3], d[2], d[1], d[0]), r.choice([torch.float32, torch.float64]), b, 1e-3)

        def payload(b0, b1):
            p.block_begin, p.block_end = b0, b1
            return dls.compress_bound(p) - _align(_align(128 + 32 * nv) + 8 * ((nb if b1 < 0 else b1) - b0 + 1))

        cut = r.randint(1, nb - 1)
        assert payload(0, -1) == payload(0, cut) + payload(cut, nb)
