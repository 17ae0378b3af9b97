"""When an access leaves its word's shadow value as it is: the rule the per-wave checker of
single traces (csrc/hr_runs.cu, absorbs()) reads off the FSM table's index, restated here and
compared with the whole step on every shadow value reachable in small grids."""
import pytest

from tests.test_fsm_table import _step_pow2, table  # noqa: F401

ACCS = [(tid, op) for tid in range(8) for op in range(3)]
CLOCKS = [(0, 0), (0, 1), (1, 0), (1, 1)]


def rule(t, o, tid, op, bc, wc, ktag, bd, ws):
    """(unchanged, unchanged for every thread) by the table index alone."""
    state, hi = o >> 59, o >> 32
    if (hi >> 24) & 7 != ktag:
        return False, False
    x = tid ^ (o & 0xFFFFFFFF)
    trel = 0 if x == 0 else 3 if x >> bd else 2 if x >> ws else 1
    srel = 2 if (hi >> 8) & 0xFFFF != bc else 1 if hi & 0xFF != wc else 0
    e = int(t[(state << 6) | (op << 4) | (trel << 2) | srel])
    if e & 31 != state:
        return False, False
    level = e >> 5
    same = {1: trel == 0 and srel == 0, 2: trel <= 1 and srel == 0, 3: trel <= 2 and srel != 2}.get(level, level in (4, 5))
    return same, same and level >= 4


@pytest.mark.parametrize("bd,ws", [(2, 1), (1, 1), (2, 0)])
def test_rule_equals_step_on_every_reachable_value(table, bd, ws):  # noqa: F811
    t, _ = table
    seen, frontier = {0}, [0]
    while frontier:
        nxt = {_step_pow2(t, s, *a, *c, k, bd, ws) for s in frontier for a in ACCS for c in CLOCKS for k in (0, 1)}
        frontier = list(nxt - seen)
        seen |= nxt
    assert len(seen) > 100
    for s in seen:
        for k in (0, 1):
            for bc, wc in CLOCKS:
                for a in ACCS:
                    same, every = rule(t, s, *a, bc, wc, k, bd, ws)
                    assert same == (s != 0 and _step_pow2(t, s, *a, bc, wc, k, bd, ws) == s)
                    if every:  # from any thread, in any later wave of the kernel
                        assert all(_step_pow2(t, s, b, a[1], *c, k, bd, ws) == s for b in range(8) for c in CLOCKS)
