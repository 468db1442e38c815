"""The end of a producer that gives up: which phase of which barrier it waits for (csrc/pt_sm100_ptx.cuh, drain_ring)."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_09290_b200", "csrc")


class Barrier:
    """One mbarrier that completes a phase per fill; waiting for the parity of the phase before the current one succeeds at once."""

    def __init__(self):
        self.phase = 0

    def try_wait(self, parity):
        return (self.phase & 1) != parity


def drain_waits(full, stages, issued):
    """The (stage, parity) pairs drain_ring waits for."""
    return [(i % stages, (i // stages) & 1) for i in range(max(0, issued - stages), issued)]


def test_the_drain_waits_for_exactly_the_copies_in_flight():
    for stages in range(1, 9):
        for issued in range(0, 4 * stages + 3):
            for landed in range(max(0, issued - stages), issued + 1):            # uses [0, landed) have arrived
                ring = [Barrier() for _ in range(stages)]
                for i in range(landed):
                    ring[i % stages].phase += 1
                waits = drain_waits(ring, stages, issued)
                blocked = {s for s, parity in waits if not ring[s].try_wait(parity)}
                assert blocked == {i % stages for i in range(landed, issued)}


def test_every_producer_that_gives_up_drains_by_phase():
    for name in ("pt_conv_sm100.cu", "pt_bn.cu", "pt_gate.cu"):
        src = open(os.path.join(CSRC, name)).read()
        # a wait for either parity succeeds at once, whatever is in flight
        assert not re.search(r"try_wait\([^;]*, 0\) && !\S*try_wait\([^;]*, 1\)", src), name
        assert "drain_ring(" in src, name
