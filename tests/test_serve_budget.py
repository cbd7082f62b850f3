"""The server's budget counts what its slots hold (CPU only): reserved workspaces
are off it from the start, requests count with what they need beyond theirs, and
no request is refused for a reservation."""
from paper_2203_02798_gb300.serve import SLOT_WORKSPACE, Request, Scheduler, run_trace, slot_workspace

GB = 1 << 30


def test_reserved_bytes_are_off_the_budget():
    s = Scheduler(slots=4, hbm_budget=10 * GB, slot_bytes=GB)
    for i, f in enumerate([GB // 2, 3 * GB, 5 * GB, GB]):      # beyond a slot's GB: 0, 2, 4, 0
        assert s.arrive(Request(i, 0.0, f))
    started = s.admit()
    assert [r.rid for r in started] == [0, 1, 2, 3] and s.used == 6 * GB   # 4 + 6 of 10 GB
    assert s.arrive(Request(4, 0.0, 2 * GB))
    s.release(started[0])
    assert s.admit() == []                                     # 4 + 6 + 1 > 10: a slot is free, the memory is not
    s.release(started[1])
    assert [r.rid for r in s.admit()] == [4]
    assert not s.arrive(Request(5, 0.0, 8 * GB))               # 4 + 7 > 10: never fits


def test_the_reservation_gives_way_to_requests_and_small_budgets():
    def plan(footprints, slots, budget):
        return slot_workspace([Request(i, 0.0, f) for i, f in enumerate(footprints)], slots, budget)
    assert plan([10 << 20], 8, 150 * 10 ** 9) == SLOT_WORKSPACE
    assert plan([10 << 20], 8, 7 * GB) == 0                    # eight slots' GB do not fit
    assert plan([143 * 10 ** 9], 8, 150 * 10 ** 9) == 0        # fits the budget, but not beside the reservations
    assert plan([143 * 10 ** 9], 4, 150 * 10 ** 9) == SLOT_WORKSPACE
    assert plan([160 * 10 ** 9, 1], 8, 150 * 10 ** 9) == SLOT_WORKSPACE   # rejected in any case
    assert plan([], 2, 3 * GB) == SLOT_WORKSPACE


def test_every_request_that_fits_the_budget_is_served():
    budget = 12 * GB
    for footprints in ([12 * GB, GB], [5 * GB] * 6, [GB // 4] * 20):
        reqs = [Request(i, 0.0, f) for i, f in enumerate(footprints)]
        held = slot_workspace(reqs, 4, budget)
        done, rejected = run_trace(reqs, lambda slot, r: r.rid, 4, budget, slot_bytes=held)
        assert not rejected and len(done) == len(reqs)
