"""Failure model of the projection that walks x (csrc/evx_nn_tc.cu): planes alternate between two
buffers with an mbarrier each, loaded two ahead. A bounded wait that runs out at any plane must
leave no copy in flight that the CTA has not waited for, start no copy into a buffer that one
may still be filling."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_21748_gb300", "csrc")


def walk(units, late):
    """Planes per unit; the wait for plane number `late` runs out. Returns the drained planes."""
    k, in_flight = 0, set()

    def load(n):
        assert not any(m % 2 == n % 2 for m in in_flight), "copy into a buffer still being filled"
        in_flight.add(n)

    for planes in units:
        load(k)
        load(k + 1)
        for q in range(planes):
            if k == late:
                drained = {k + m for m in range(2) if q + m < planes}
                assert in_flight == drained
                return drained
            in_flight.discard(k)
            if q + 2 < planes:
                load(k + 2)
            k += 1
    assert not in_flight
    return set()


@pytest.mark.parametrize("units", [[3], [4, 3], [10, 3, 18]])
def test_every_late_plane_is_drained(units):
    for late in range(sum(units) + 1):
        assert (late in walk(units, late)) == (late < sum(units))


def test_no_bounded_wait_is_ignored():
    """The result of a bounded pipeline wait is used, or its mark is: the projection reads the
    flag after the plane's barrier, guards the loads and stores after it, and drains at its end."""
    with open(os.path.join(CSRC, "evx_nn_tc.cu")) as f:
        text = f.read()
    dropped = re.findall(r"(?m)^\s*(?:\(void\))?ring_wait(?:_long)?\((.*)\);", text)
    assert all(args.endswith("(int)k + 1") for args in dropped), dropped
    i = text.index("project_walk_kernel(const")
    body = text[i:text.index("// =", i)]
    order = ["(int)k + 1", "__syncthreads();  // the plane", "mark = *abort_flag", "if (go && q + 2 < np) load(", "if (go && q >= 2)",
             "r.out[", "if (!go && threadIdx.x == 0)", "tc_wait("]
    at = [body.index(o) for o in order]
    assert at == sorted(at) and body.count("r.out[") == 1 and "nunits && go;" in body


def test_every_thread_takes_the_same_way():
    """A thread reads the flag some time after plane k's barrier; by then threads ahead of it may
    have marked plane k + 1 (not k + 2: they wait for it at the barrier between)."""
    for k in range(6):
        for first in [None] + list(range(8)):  # plane whose wait ran out first
            seen = set()
            for ahead in (0, 1):
                flag = first + 1 if first is not None and first <= k + ahead else 0
                seen.add(flag == 0 or flag > k + 1)
            assert seen == {first is None or first > k}
