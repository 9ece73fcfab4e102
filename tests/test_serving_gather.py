"""The hold before a group's first tick (BatchedServer, gather_s) on the CPU, with stand-in systems.

A hold pays when a request joins in time: one that is due and can be admitted shares the
first tick. It must not cost time where none can: requests kept out by the budget, by a
larger request at the head of the queue or by their own arrival after a tick of the group
delay nobody. gather_s is made long against the work, so that a hold that runs out shows.
"""
import time

import pytest

from paper_1905_01348_gb300.serve import BatchedServer, Request


class Tick:
    """A system whose step takes step_s."""

    def __init__(self, req, slot, step_s=0.003):
        self.req, self.step_s, self.k = req, step_s, 0

    def step(self):
        time.sleep(self.step_s)
        self.k += 1
        return 0, {"energy": float(self.k), "dipole": [0.0, 0.0, 0.0], "scf_iters": 1}

    def close(self):
        pass


class Together:
    """Steps its members one after another; records who was batched with whom."""
    made = []

    def __init__(self, systems):
        self.systems = list(systems)
        Together.made.append(tuple(s.req.rid for s in self.systems))

    def step(self):
        return 0, [s.step()[1] for s in self.systems]

    def close(self):
        pass


def serve(reqs, budget, gather_s, sizes=None, step_s=None, **more):
    Together.made.clear()
    srv = BatchedServer(lambda r: (sizes or {}).get(r.rid, 1), lambda r, s: Tick(r, s, (step_s or {}).get(r.rid, 0.003)),
                        Together, budget_bytes=budget, gather_s=gather_s, **more)
    outs = srv.run(reqs)
    assert all(o.error is None and len(o.energy) == r.steps for r, o in zip(reqs, outs))
    return srv, outs


def test_requests_due_within_the_hold_share_the_first_tick():
    serve([Request(0, "si8", 3, 0.0), Request(1, "si8", 3, 0.05)], budget=10, gather_s=2.0, max_active=4)
    assert Together.made[0] in ((0, 1), (1, 0))


def test_a_lone_request_is_not_held():
    srv, _ = serve([Request(0, "si8", 3, 0.0)], budget=10, gather_s=5.0, max_active=4)
    assert srv.wall_s < 2.0


@pytest.mark.parametrize("reserve", [0, 2])
def test_requests_kept_out_by_the_budget_hold_nobody(reserve):
    """Room for one request at a time: every request of the group is due, none can join."""
    srv, _ = serve([Request(k, "si8", 3, 0.0) for k in range(6)], budget=1 + reserve, gather_s=5.0, max_active=4,
                   group_reserve=lambda key: reserve)
    assert srv.wall_s < 4.0 and srv.peak_batch == 1


def test_a_request_behind_a_larger_one_holds_nobody():
    """Admission is in arrival order: 3 would fit, but waits behind 2, which waits for 0."""
    reqs = [Request(0, "si216", 100, 0.0), Request(1, "si8", 3, 0.0), Request(2, "si64", 3, 0.0),
            Request(3, "si8", 3, 0.0)]
    _, outs = serve(reqs, budget=10, gather_s=5.0, sizes={0: 6, 1: 1, 2: 6, 3: 1}, step_s={0: 0.02}, max_active=4)
    assert outs[1].finished_s < 1.5 < outs[0].finished_s


def test_requests_further_apart_than_a_tick_are_not_held():
    """A request that starts at once keeps a later one waiting for a tick at most, so a group
    that knows the length of its ticks holds no longer than one."""
    reqs = [Request(0, "si8", 3, 0.0)] + [Request(k, "si8", 3, 1.5 + 0.5 * k) for k in range(1, 4)]
    _, outs = serve(reqs, budget=10, gather_s=1.0, max_active=4)
    for r, o in zip(reqs, outs):
        assert o.finished_s - r.arrival_s < 0.4
