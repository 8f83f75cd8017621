"""The plan of a one-launch grad_W + grad_X, without a GPU: every unit of both products is some pair's, exactly once.

The order in which a pair takes units is restated here from the header's description of the plan's numbers.
"""
import random

import pytest

from paper_2409_09099_b200 import binding as B, build


@pytest.fixture(scope="module", autouse=True)
def lib():
    build.build()
    return B.load()


def _shapes():
    rng = random.Random(7)
    some = [(128, 128, 128), (256, 256, 512), (768, 768, 8192), (3072, 768, 8192), (768, 3072, 8192), (3840, 1280, 16384),
            (1280, 5120, 16384), (11008, 4096, 16384), (50304, 768, 1024)]
    return some + [tuple(128 * rng.randint(1, 86) for _ in range(3)) for _ in range(60)]


def _units_of(pair, pairs, late, early, early_first, n):
    """grad_X units of one pair in its order."""
    n_early = pairs - late
    is_late = pair < late
    rank = (n_early + pair if is_late else pair - late) if early_first else pair
    got = [] if is_late else [r * n_early + pair - late for r in range(early)]
    got += range(early * n_early + rank, n, pairs)
    return [u for u in got if u < n]


@pytest.mark.parametrize("dt", [B.BF16, B.E5M2])
@pytest.mark.parametrize("sms", [148, 20])
def test_every_unit_once(dt, sms):
    for O, I, T in _shapes():
        for ws in (None, B.load().sste_workspace_bytes()):
            bw, splits, split_from, gw, bx, gx, pairs, late, early, ef, sx, w_sum = B.joint_plan(dt, O, I, T, sms, ws)
            elt = 2 if dt == B.BF16 else 1
            wt, xt = -(-O // 256) * -(-I // bw), -(-T // 256) * -(-I // bx)
            assert bw in (128, 256) and bx in (128, 256) and 1 <= pairs <= sms // 2 and 0 <= late <= pairs
            assert 1 <= gw <= -(-O // 256) and 1 <= gx <= -(-T // 256)
            w_units = split_from + (wt - split_from) * splits
            if splits > 1:
                assert ws is None and -(-T // (256 // elt)) // splits >= (2 if w_sum else 8) and split_from % pairs == 0
            else:
                assert split_from == wt
            assert late == w_units % pairs or (late == pairs and w_units % pairs == 0)   # pairs with a unit more come first
            if w_sum:                                # sums only where all ranges run at once
                assert ws is None and split_from == 0 and splits > 1 and wt * splits <= sms // 2
            if sx > 1:
                assert ws is None and wt * splits + xt * sx <= sms // 2 and -(-O // (128 // elt)) // sx >= 2
            seen = sorted(u for p in range(pairs) for u in _units_of(p, pairs, late, early, ef, xt * sx))
            assert seen == list(range(xt * sx)), (O, I, T)
