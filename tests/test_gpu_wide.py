"""The wide-band kernel (batched and served pairs whose band has outgrown one
CTA) against the oracle, at the edges of its passes: tiles of one and of
several strips, groups of one and of several CTAs, block lengths that do not
divide the segments, strings at every alignment, ends reached early (unequal
lengths, one symbol), and slides that outrun their warp.  Integer results: the
tolerance is zero."""
import time

import numpy as np
import pytest

from gpu_util import dev
from paper_2306_17461_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _gap_pair(n, k, gap, extra):
    """k edits in the first half of n characters and k in the second, with an
    unedited stretch of `gap` between: one slide of about that length."""
    rng = W.rng_for(301, extra)
    sym = W.Symbols(4)
    A = sym.draw(rng, n + gap)
    pos = np.concatenate([rng.choice(n // 2, k, replace=False), n // 2 + gap + rng.choice(n // 2, k, replace=False)])
    return A, W.plant(rng, A, np.sort(pos), sym)


def _pairs():
    rng = np.random.default_rng(302)
    out = []
    for n, k, sigma in [(30_000, 2300, 4), (30_000, 2600, 64), (60_001, 4200, 2), (24_000, 3100, 256)]:
        out.append(W.random_pair(rng, n, k, sigma))
    out.append((rng.integers(0, 4, 9001, dtype=np.uint8), rng.integers(0, 4, 9500, dtype=np.uint8)))  # unrelated
    out.append((rng.integers(0, 4, 5000, dtype=np.uint8), rng.integers(4, 8, 5003, dtype=np.uint8)))  # disjoint
    out.append((np.zeros(3000, np.uint8), np.zeros(9000, np.uint8)))  # one symbol, unequal lengths
    A, B = W.random_pair(rng, 20_000, 300, 4)
    out.append((A, B[: B.size - 4000]))  # a long end gap
    out.append((A[5000:], B))            # and one at the start
    out.append(_gap_pair(20_000, 1500, 150_000, 1))
    p = W.lcp_length_pair(9000, 0.9, n=100_000)
    out.append((p.A, p.B))
    return out


@pytest.fixture(scope="module")
def pairs(orc):
    ps = _pairs()
    return ps, orc.many("lv", ps)


@pytest.mark.parametrize("cfg", [{}, {"grid_ctas": 1}, {"grid_ctas": 3, "block_rounds": 5},
                                 {"grid_ctas": 5, "block_rounds": 64}, {"block_rounds": 1}, {"warp_cap": 512}],
                         ids=["default", "one_cta", "g3_h5", "g5_h64", "h1", "cap512"])
def test_wide_bands_match_oracle(pairs, cfg):
    from paper_2306_17461_gb300 import binding as ed

    ps, want = pairs
    assert sum(int(k) > 2048 for k in want) >= 9  # past the batch kernel's band
    dA, dB = [], []
    for i, (A, B) in enumerate(ps):  # strings at odd offsets of their buffers
        oa, ob = i % 5, (3 * i + 1) % 7
        dA.append(dev(np.concatenate([np.full(oa, 9, np.uint8), A]))[oa:])
        dB.append(dev(np.concatenate([np.full(ob, 9, np.uint8), B]))[ob:])
    with ed.Context(device=0, **cfg) as c:
        got = ed.ed_distance_batch_dev(c.h, dA, dB)
        assert np.array_equal(got, want), cfg
        again = ed.ed_distance_batch_dev(c.h, dB, dA)  # the strings exchanged
        assert np.array_equal(again, want), cfg


@pytest.mark.parametrize("call", ["batch", "served"])
@pytest.mark.parametrize("h", [32, 5, 64])
def test_round_cap(orc, h, call):
    """max_rounds counts whole blocks of h rounds from round 0, wherever the
    batch kernel left the pair: a cap that ends the block holding round k
    gives the distance, one less is refused."""
    from paper_2306_17461_gb300 import binding as ed

    A, B = W.random_pair(np.random.default_rng(304), 24_000, 3100, 256)
    k = orc.lv(A, B)
    assert k > 2048
    cap = (k // h + 1) * h - 1
    for rounds in (cap, cap - 1, 2080):
        with ed.Context(device=0, block_rounds=h, max_rounds=rounds) as c:
            try:
                if call == "batch":
                    got = int(ed.ed_distance_batch_dev(c.h, [dev(A)], [dev(B)])[0])
                else:
                    t, st = ed.ed_submit(c.h, A, B), ed.ED_EAGAIN
                    while st == ed.ED_EAGAIN:
                        st, got = ed.ed_poll(c.h, t)
                        time.sleep(0.001)
            except ed.EdError as e:
                got = e.code
        assert got == (k if rounds == cap else ed.ED_ELIMIT), rounds
