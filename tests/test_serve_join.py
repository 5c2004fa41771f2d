"""Live serving: for which setups an idle driver with one ready request waits."""
from paper_2403_11636_gb300.serve import BatchServer, Request
from tests.test_serve import LiveFP, make_live_fakes


def serve(specs, join_s):
    """specs: (footprint, setup seconds, arrival); two cycles of 20 ms each."""
    setup, cycle, release, st = make_live_fakes(cycle_dur=0.02)
    reqs = []
    for k, (fp, dur, t) in enumerate(specs):
        p = LiveFP(k, fp, 2)
        p.dur = dur
        reqs.append(Request(k, p, t))
    res = BatchServer(setup, None, release, lambda p: p.fp, budget_bytes=1e4, slots=8, cycle_fn=cycle,
                      join_s=join_s).run(reqs)
    return res, st["cycles"]


def test_no_wait_for_a_setup_that_takes_longer():
    """The other request is 40 times as large: its setup cannot end in time."""
    res, cycles = serve([(10, 0.05, 0.0), (400, 1.0, 0.0)], join_s=0.5)
    assert cycles[0] == [0] and res[0].finished < 0.4


def test_waits_for_a_like_setup():
    res, cycles = serve([(10, 0.05, 0.0), (10, 0.05, 0.03)], join_s=0.5)
    assert cycles[0] == [0, 1]


def test_no_wait_without_join():
    res, cycles = serve([(10, 0.05, 0.0), (10, 0.05, 0.03)], join_s=0.0)
    assert cycles[0] == [0]


def test_join_is_the_callers_choice():
    assert BatchServer.gpu(live=True, join_s=0.0).join_s == 0.0
    assert BatchServer.gpu(live=True).join_s == 0.03
