"""bench.py's burst figures are the device's: a step counts only if it was enqueued before the spin in front of it had ended."""
import pytest

from bench import enqueued_ahead


class Device:
    """A stream whose spin ends after `cycles` and a host that takes `host` cycles to enqueue a step."""

    def __init__(self, host):
        self.host, self.spins, self.idles = host, [], 0

    def idle(self):
        self.idles += 1

    def spin(self, cycles):
        self.spins.append(cycles)

    def enqueue(self):
        return self

    def query(self):                 # has the event behind the spin passed?
        return self.spins[-1] <= self.host


@pytest.mark.parametrize("host,spins", [(0, [200_000]), (199_999, [200_000]), (200_000, [200_000, 400_000]), (1_000_000, [200_000, 400_000, 800_000, 1_600_000])])
def test_a_step_enqueued_too_late_is_repeated_behind_a_longer_spin(host, spins):
    d = Device(host)
    assert enqueued_ahead(d.idle, d.spin, d.enqueue) is True
    assert d.spins == spins and d.idles == len(spins)


def test_a_host_that_is_never_ahead_is_reported():
    d = Device(10**12)
    assert enqueued_ahead(d.idle, d.spin, d.enqueue) is False
    assert len(d.spins) == 6 and d.spins[-1] < 10_000_000      # (some milliseconds: no wait grows without bound)
