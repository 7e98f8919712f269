"""Failure detection without a GPU fault.

* Every device-side wait of the tile kernel is bounded by %globaltimer.
  With a bound of 1 ns a wait that cannot be answered at once gives up: the
  kernel records where (site, CTA, round), every CTA leaves, and the host
  returns ED_ETIMEOUT with that record.  The pair used makes such a wait
  certain: tiles beyond the band skip ahead and then wait for their inner
  neighbour to compute about a thousand rounds.  The device stays usable: a
  context with the default bound computes the exact distance on the same
  strings.
* Host-side refusals: a memory budget too small for the strings returns
  ED_ENOMEM before anything is allocated, and serving refuses admission
  (ED_EBUSY) when the arena cannot hold a request while another one is
  resident, then admits it once that one has retired."""
import re
import time

import pytest

from gpu_util import dev
from paper_2306_17461_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.timeout(300)
def test_bounded_wait_gives_up_and_the_device_stays_usable(orc):
    from paper_2306_17461_gb300 import binding as ed

    # thousands of rounds over the whole grid
    p = W.make_pair(51, 1_000_000, 3000, sigma=4)
    want = orc.lv(p.A, p.B)
    dA, dB = dev(p.A), dev(p.B)
    c = ed.Context(device=0, spin_limit_ns=1)
    try:
        with pytest.raises(ed.EdError) as ei:
            c.distance_dev(dA, dB)
        assert ei.value.code == ed.ED_ETIMEOUT, str(ei.value)
        m = re.search(r"kernel check failed: site (\d+) cta (\d+) t (\d+)", str(ei.value))
        assert m, str(ei.value)
        # 1 job close, 2 group barrier, 3 idle CTA, 4 neighbours' edge words, 5 epoch barrier
        assert 1 <= int(m.group(1)) <= 5
    finally:
        c.close()
    c2 = ed.Context(device=0)
    try:
        assert c2.distance_dev(dA, dB) == want
    finally:
        c2.close()


def test_budget_too_small_for_the_strings():
    import numpy as np

    from paper_2306_17461_gb300 import binding as ed

    c = ed.Context(device=0, mem_budget_bytes=1 << 20)
    try:
        A = np.zeros(2 << 20, np.uint8)
        with pytest.raises(ed.EdError) as ei:
            c.distance(A, A)
        assert ei.value.code == ed.ED_ENOMEM
    finally:
        c.close()


@pytest.mark.timeout(300)
def test_serving_refuses_admission_on_memory_then_admits(orc):
    from paper_2306_17461_gb300 import binding as ed

    # arena: half of a 200 MB budget; a resident 2 x 30 MB pair leaves no room
    # for a second one
    big = W.make_pair(52, 30_000_000, 30_000, sigma=4)
    small = W.make_pair(53, 30_000_000, 10, sigma=4)
    want_big, want_small = orc.lv(big.A, big.B, nthreads=8), orc.lv(small.A, small.B)
    c = ed.Context(device=0, mem_budget_bytes=200 << 20, max_inflight=64)
    try:
        t1 = ed.ed_submit(c.h, big.A, big.B)
        with pytest.raises(ed.EdError) as ei:
            ed.ed_submit(c.h, small.A, small.B)
        assert ei.value.code == ed.ED_EBUSY
        # admitted once the first request has retired and freed its memory
        t2 = None
        k1 = None
        deadline = time.time() + 240
        while t2 is None and time.time() < deadline:
            st, k = ed.ed_poll(c.h, t1)
            if st == ed.ED_OK:
                k1 = k
            try:
                t2 = ed.ed_submit(c.h, small.A, small.B)
            except ed.EdError as e:
                assert e.code == ed.ED_EBUSY
                time.sleep(0.01)
        assert t2 is not None
        while k1 is None:
            st, k = ed.ed_poll(c.h, t1)
            if st == ed.ED_OK:
                k1 = k
            time.sleep(0.002)
        while True:
            st, k2 = ed.ed_poll(c.h, t2)
            if st == ed.ED_OK:
                break
            time.sleep(0.002)
        assert (k1, k2) == (want_big, want_small)
        assert ed.ed_serve_counters(c.h)["admitted"] == 2
    finally:
        c.close()


def test_slots_new_in_a_failed_call_are_cleared(orc):
    """A call that fails after the job slots have grown (no room for the edge
    words that come next) leaves slots that were never cleared; the next call
    must not take what lies in them for answers.  The memory they land in holds
    words that read as "no mismatch" of the first jobs."""
    import torch

    from paper_2306_17461_gb300 import binding as ed

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    keep, gf = 4 * (2 * 600_000 + 5), 8 * (2 * 2048 * sms + 5)  # of a pair of 600 thousand characters
    slots, edges = 2 * sms * 33_024, 2048 * sms
    short, mid, far, last = (W.make_pair(140 + i, n, k, sigma=4)
                             for i, (n, k) in enumerate([(1500, 4), (600_000, 2), (4_000_000, 2), (300_000, 2)]))
    with ed.Context(device=0, mem_budget_bytes=keep + gf + slots + edges * 5 // 8) as c:
        assert c.distance_dev(dev(short.A), dev(short.B)) == orc.lv(short.A, short.B)
        bufs = [(dev(p.A), dev(p.B)) for p in (mid, far, last)]
        words = (torch.arange(8 << 20, device="cuda") % 8 + 1) << 32 | 0xFFFFFFFF
        torch.cuda.synchronize()
        del words
        torch.cuda.empty_cache()
        for a, b in bufs[:2]:  # no room for the edge words, then for the frontier (which gives its room back)
            with pytest.raises(ed.EdError) as ei:
                c.distance_dev(a, b)
            assert ei.value.code == ed.ED_ENOMEM
        assert c.distance_dev(*bufs[2]) == orc.lv(last.A, last.B)
        assert c.stats()["long_slides"] >= 1


@pytest.mark.timeout(300)
@pytest.mark.parametrize("call", ["batch", "served"])
def test_wide_band_under_every_budget(orc, call):
    """A pair whose band (40001 diagonals) is wider than two of its four CTAs
    hold: whatever the memory budget, the call gives the distance or says that
    memory is short.  What the pair takes with its tiles in shared memory (job
    slots, re-tiling buffers, the batch kernel's frontier, edges and control
    words) is enough."""
    from paper_2306_17461_gb300 import binding as ed

    n = 20_000
    rng = W.rng_for(303, 0)
    A, B = W.Symbols(4).draw(rng, n), W.Symbols(4).draw(rng, n) + 4
    want = orc.lv(A, B)
    assert 2 * want + 1 > 2 * 16_384
    dA, dB = dev(A), dev(B)
    enough = 4 * 2 * 33_024 + 16 * (n + 5) + 4 * 4_099 + 4 * 2_048 + 8 * 4_096
    base = 0 if call == "batch" else 64 << 20  # the arena's smallest size
    short = 0
    for budget in list(range(64 << 10, enough, 48 << 10)) + [enough + i * (48 << 10) for i in range(12)]:
        with ed.Context(device=0, grid_ctas=4, mem_budget_bytes=base + budget) as c:
            try:
                if call == "batch":
                    k = int(ed.ed_distance_batch_dev(c.h, [dA], [dB])[0])
                else:
                    ticket = ed.ed_submit(c.h, A, B)
                    st = ed.ED_EAGAIN
                    while st == ed.ED_EAGAIN:
                        st, k = ed.ed_poll(c.h, ticket)
                        time.sleep(0.001)
                assert k == want, budget
            except ed.EdError as e:
                assert e.code == ed.ED_ENOMEM and budget < enough, (budget, str(e))
                short += 1
    assert short > 0
