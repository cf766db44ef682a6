"""A CPU model of the stream kernel's ring with one and two compactor teams (host logic, no GPU): a producer fills the ring's stages in order, the
teams take the chunks in turn, read a stage and write an operand set, the MMA issuer reads both and releases them with commits that land
some time later.  Barriers as in `test_issuer_protocol_model`: a waiter sees a phase's parity only.  The model fails on a wait that
passes on a stage or set that does not hold the chunk the waiter expects, on over-arrival and on a state in which nobody can move.

It pins the rule the kernel follows: a ring of odd depth, whose stages go to two teams in turn, has a full barrier per stage AND team; with one per
stage a team skips every second phase, and a wait can pass on an earlier one."""
import random

import pytest

from test_issuer_protocol_model import Bar, Ring


def simulate(chunks, depth, sets, teams, per_team, seed):
    rnd = random.Random(seed)
    n_full = 2 * depth if teams == 2 and depth % 2 and per_team else depth
    full = [Bar(f"full{i}", 1) for i in range(n_full)]
    free = [Bar(f"free{i}", 2) for i in range(depth)]         # a team, and the commit
    aready = [Bar(f"aready{i}", 1) for i in range(sets)]
    afree = [Bar(f"afree{i}", 1) for i in range(sets)]
    holds, operands = [None] * depth, [None] * sets
    landing, commits = [], []

    def producer():
        rp, rf = Ring(), Ring()
        for g in range(chunks):
            if rp.wrapped:
                while not free[rp.s].passed(rp.par ^ 1):
                    yield
            landing.append((full[rf.s], rp.s, g))
            rp.adv(depth)
            rf.adv(n_full)
            yield

    def team(t):
        rf, rs = Ring(), Ring()
        for g in range(chunks):
            if g % teams == t:
                while not full[rf.s].passed(rf.par):
                    yield
                if holds[rf.s % depth] != g:
                    raise RuntimeError(f"team {t} passed a stale phase: the stage holds chunk {holds[rf.s % depth]}, not {g}")
                while rs.wrapped and not afree[rs.s].passed(rs.par ^ 1):
                    yield
                yield
                operands[rs.s] = g
                aready[rs.s].arrive(f"team{t}")
                free[rf.s % depth].arrive(f"team{t}")
            rf.adv(n_full)
            rs.adv(sets)
            yield

    def issuer():
        rf, rs = Ring(), Ring()
        for g in range(chunks):
            while not full[rf.s].passed(rf.par):
                yield
            while not aready[rs.s].passed(rs.par):
                yield
            if holds[rf.s % depth] != g or operands[rs.s] != g:
                raise RuntimeError(f"the issuer passed a stale phase: chunks {holds[rf.s % depth]} and {operands[rs.s]}, not {g}")
            commits.append((afree[rs.s], g))
            commits.append((free[rf.s % depth], g))
            rf.adv(n_full)
            rs.adv(sets)
            yield

    agents = {"producer": producer(), "issuer": issuer(), **{f"team{t}": team(t) for t in range(teams)}}
    slow = rnd.choice([None, None] + sorted(agents))          # one agent may be far behind the others
    idle = 0
    while agents:
        moved = False
        if commits and rnd.random() < 0.5:
            commits.pop(0)[0].arrive("a commit")
            moved = True
        while landing and rnd.random() < 0.5:
            bar, stage, g = landing.pop(rnd.randrange(len(landing)))
            holds[stage] = g
            bar.arrive("a load")
            moved = True
        names = list(agents)
        rnd.shuffle(names)
        before = tuple((b.phase, b.pending) for b in full + free + aready + afree)
        for n in names:
            if n == slow and rnd.random() < 0.9:
                moved = True
                continue
            try:
                next(agents[n])
            except StopIteration:
                del agents[n]
                moved = True
        moved = moved or tuple((b.phase, b.pending) for b in full + free + aready + afree) != before
        idle = 0 if moved or commits or landing else idle + 1
        if idle > 200:
            raise RuntimeError(f"deadlock: {sorted(agents)} cannot move")


@pytest.mark.parametrize("teams,sets", [(1, 2), (2, 2), (2, 4)])
@pytest.mark.parametrize("depth", [1, 2, 3, 4, 5, 6])
def test_every_depth_is_safe(depth, teams, sets):
    for seed in range(150):
        simulate(random.Random(seed).randint(1, 40), depth, sets, teams, True, seed)


@pytest.mark.parametrize("depth", [3, 5])
def test_one_full_barrier_per_stage_of_an_odd_ring_is_not(depth):
    failures = 0
    for seed in range(300):
        try:
            simulate(40, depth, 4, 2, False, seed)
        except RuntimeError as e:
            assert "stale phase" in str(e) or "deadlock" in str(e) or "over-arrival" in str(e)
            failures += 1
    assert failures > 0
