"""Host logic of the paired GEMM's early stop: whatever the two CTAs had issued when they stopped, every stage's barrier
completes after what is owed to it has been given, once all copies have landed and not before (a model of the barriers,
counts of arrivals and bytes per phase)."""
import ctypes

import pytest

NOTHING, COPIES, ARRIVAL, BYTES = range(4)


class Barrier:
    """One arrival per phase; a phase completes at no pending arrival and no bytes outstanding."""

    def __init__(self):
        self.phase, self.pending, self.bytes = 0, 1, 0

    def _settle(self):
        if self.pending == 0 and self.bytes == 0:
            self.phase, self.pending = self.phase + 1, 1

    def arrive_expect(self, n):
        self.bytes += n
        self.pending -= 1
        assert self.pending >= 0
        self._settle()

    def complete(self, n):
        self.bytes -= n
        self._settle()

    def passed(self, parity):
        """What a wait for `parity` sees."""
        return (self.phase & 1) != parity


@pytest.fixture(scope="module")
def landing():
    from paper_2601_03700_gb300 import build
    build.build()
    import paper_2601_03700_gb300 as adept
    f = adept.load_library().adept_debug_pair_landing
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    f.restype = None

    def call(n0, n1, stages):
        out = (ctypes.c_int * (2 * stages))()
        f(n0, n1, stages, out)
        return [(out[2 * s], out[2 * s + 1]) for s in range(stages)]
    return call


@pytest.mark.parametrize("stages", [1, 2, 6, 10])
def test_every_stage_completes_after_its_last_copy(landing, stages):
    for n0 in range(3 * stages + 2):
        for n1 in range(max(0, n0 - stages), n0 + stages + 1):
            bars = [Barrier() for _ in range(stages)]
            for k in range(min(n0, n1)):        # sent by both
                bars[k % stages].arrive_expect(2)
                bars[k % stages].complete(1)
                if k + stages < max(n0, n1):    # consumed: its last copy has landed
                    bars[k % stages].complete(1)
            late = {k % stages: 1 for k in range(max(0, max(n0, n1) - stages), min(n0, n1))}
            for k in range(min(n0, n1), max(n0, n1)):
                if k < n0:
                    bars[k % stages].arrive_expect(2)
                late[k % stages] = 1            # the one copy under way
            for s, (owe, parity) in enumerate(landing(n0, n1, stages)):
                if s >= max(n0, n1):
                    assert owe == NOTHING
                    continue
                if owe == ARRIVAL:
                    bars[s].arrive_expect(1)
                elif owe == BYTES:
                    bars[s].complete(1)
                else:
                    assert owe == COPIES
                assert not bars[s].passed(parity), (n0, n1, s)
                bars[s].complete(late[s])
                assert bars[s].passed(parity) and bars[s].bytes == 0, (n0, n1, s)
