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
    """A bounded pipeline wait that is a statement of its own drops its result; after a failed
    one the projection drains before it could load or store again."""
    with open(os.path.join(CSRC, "evx_nn_tc.cu")) as f:
        text = f.read()
    assert not re.findall(r"(?m)^\s*(?:ring_wait|ring_wait_long)\(.*\);", text)
    body = text[text.index("project_walk_kernel(const"):text.index("// =", text.index("project_walk_kernel(const"))]
    stop = body.index("__syncthreads_or(!arrived)")
    assert stop < body.index("tc_wait(") < body.index("load(q + 2") < body.index("r.out[")
