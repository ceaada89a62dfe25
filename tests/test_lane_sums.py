"""The error bounds of the search's shared distances, pinned by emulating their
arithmetic in IEEE single precision against exact rational sums (csrc/search.cu):

* a row summed by G lanes, four sums each, joined by a butterfly: every term
  takes at most ceil(chunks / G) + 4 + log2 G roundings (lane_rel_bound holds
  six more);
* the float-float distance of one warp: within the (3 d + 13) 2^-48 of one
  chain (ff_bound);
* the list's thresholds kc (1 -+ E2) -+ A2: a key beyond them has an interval
  apart from the point's."""
from fractions import Fraction

import numpy as np
import pytest

from test_ff_bound import _ff_step, _fma, f32


def _padded(x):
    return np.concatenate([x, np.zeros(-x.shape[0] % 32, np.float32)]).astype(np.float32)


def _lanes(chunks):
    return 4 if chunks <= 24 else 8 if chunks <= 64 else 32


def _lane_sum(a, b):
    a, b = _padded(a), _padded(b)
    chunks = a.shape[0] // 4
    G = _lanes(chunks)
    lane = []
    with np.errstate(over="ignore", under="ignore"):
        for s in range(G):
            acc = [f32(0)] * 4
            for c in range(s, chunks, G):
                for j in range(4):
                    t = f32(a[4 * c + j] - b[4 * c + j])
                    acc[j] = _fma(t, t, acc[j])
            lane.append(f32(f32(acc[0] + acc[1]) + f32(acc[2] + acc[3])))
        o = G // 2
        while o:
            lane = [f32(lane[i] + lane[i ^ o]) for i in range(G)]
            o //= 2
    assert len({float(v) for v in lane}) == 1  # the same value in every lane
    return lane[0], -(-chunks // G) + 4 + G.bit_length() - 1


def _ff_warp(a, b):
    a, b = _padded(a), _padded(b)
    chunks = a.shape[0] // 4
    lane = []
    with np.errstate(over="ignore", under="ignore"):
        for s in range(32):
            sh, sl = f32(0), f32(0)
            for c in range(s, chunks, 32):
                for i in range(4 * c, 4 * c + 4):
                    sh, sl = _ff_step(a[i], b[i], sh, sl)
            lane.append((sh, sl))
        for o in (16, 8, 4, 2, 1):
            new = []
            for i in range(32):
                (sh, sl), (oh, ol) = lane[i], lane[i ^ o]
                s1 = f32(sh + oh)
                bv = f32(s1 - sh)
                e = f32(f32(sh - f32(s1 - bv)) + f32(oh - bv))
                l1 = f32(f32(sl + ol) + e)
                h = f32(s1 + l1)
                new.append((h, f32(l1 - f32(h - s1))))
            lane = new
    assert len({(float(h), float(l)) for h, l in lane}) == 1
    return Fraction(float(np.float64(lane[0][0]) + np.float64(lane[0][1])))


@pytest.mark.parametrize("d", [1, 5, 24, 96, 100, 256, 300, 960])
def test_lane_and_warp_sums_stay_within_their_bounds(d):
    rng = np.random.default_rng(d)
    rows = [(rng.normal(size=d), rng.normal(size=d)),
            (np.abs(rng.normal(size=d)), np.abs(rng.normal(size=d)) * 1e-3),
            (rng.normal(size=d) * np.exp(rng.uniform(-20, 20, d)), rng.normal(size=d) * np.exp(rng.uniform(-20, 20, d))),
            (rng.integers(1, 9, d) * 2.0 ** -149, np.zeros(d))]
    for a, b in rows:
        a, b = a.astype(np.float32), b.astype(np.float32)
        exact = sum(((Fraction(float(x)) - Fraction(float(y))) ** 2 for x, y in zip(a, b)), Fraction(0))
        got, roundings = _lane_sum(a, b)
        bound = Fraction(roundings, 2 ** 24) * (1 + Fraction(1, 2 ** 16)) * exact + Fraction(4 * (d + 1), 2 ** 149)
        assert abs(Fraction(float(got)) - exact) <= bound
        bound = Fraction(3 * d + 13, 2 ** 48) * exact + Fraction(4 * d + 4, 2 ** 149)
        assert abs(_ff_warp(a, b) - exact) <= bound


@pytest.mark.parametrize("chunks,d", [(8, 1), (24, 96), (240, 960), (16384, 65536)])
def test_keys_beyond_the_thresholds_have_apart_intervals(chunks, d):
    G = _lanes(chunks)
    E = f32((chunks + G - 1) // G + 10 + G.bit_length() - 1) * f32(2.0 ** -24)
    Eabs = f32(f32(d + 1) * f32(2.0 ** -149)) * f32(4)
    E2, A2 = f32(f32(2) * E + f32(2.0 ** -22)), f32(f32(4) * Eabs)
    Ef, Af = Fraction(float(E)), Fraction(float(Eabs))
    rng = np.random.default_rng(chunks)
    for kc in np.concatenate([np.exp(rng.uniform(-90, 80, 40)), [2.0 ** -149, 2.0 ** -130, 1.0, 2.0 ** 120]]).astype(f32):
        k = Fraction(float(kc))
        for fused in (False, True):
            lo = _fma(kc, f32(1) - E2, -A2) if fused else f32(f32(kc * (f32(1) - E2)) - A2)
            hi = _fma(kc, f32(1) + E2, A2) if fused else f32(f32(kc * (f32(1) + E2)) + A2)
            below, above = np.nextafter(lo, f32(-np.inf)), np.nextafter(hi, f32(np.inf))
            if below >= 0:
                m = Fraction(float(below))
                assert m * (1 + Ef) + Af < k * (1 - Ef) - Af
            m = Fraction(float(above))
            assert m * (1 - Ef) - Af > k * (1 + Ef) + Af
