"""The consumer's greedy scan in rounds of four (csrc/prune.cu greedy_scan), restated
on Python integers against Algorithm 1's loop: every round reads the first four
live candidates' masks at once and keeps the second to fourth unless an earlier one
of the round took them out."""
import numpy as np
import pytest


def _loop(m, masks, R):
    live, kept = set(range(m)), []
    while live and len(kept) < R:
        p = min(live)
        kept.append(p)
        live = {v for v in live if v != p and not (masks[p] >> v) & 1}
    return kept


def _rounds(m, masks, R):
    live, kept = (1 << m) - 1, []
    while len(kept) < R and live:
        rest, p = live, []
        for _ in range(4):
            p.append((rest & -rest).bit_length() - 1 if rest else 0)  # past the last live one: rank 0
            rest &= rest - 1 if rest else 0
        for q in p:
            if len(kept) < R and (live >> q) & 1:
                kept.append(q)
                live &= ~(masks[q] | (1 << q))
    return kept


@pytest.mark.parametrize("m", [0, 1, 2, 3, 4, 5, 63, 64, 65, 127, 128])
@pytest.mark.parametrize("density", [0.0, 0.02, 0.2, 0.9, 1.0])
def test_rounds_of_four_keep_what_the_loop_keeps(m, density):
    rng = np.random.default_rng(m * 10 + int(density * 10))
    for R in (1, 2, 3, 5, 32, 64, 2**31 - 1):
        for _ in range(20):
            masks = []
            for p in range(max(m, 1)):
                bits = rng.random(128) < density  # bits of earlier ranks and past m are harmless
                masks.append(int("".join("1" if b else "0" for b in bits), 2))
            assert _rounds(m, masks, R) == _loop(m, masks, R)
