"""The bandwidths of the benchmark line: a time of several steps per launch is not
turned into one, since the state crosses memory once per launch."""
from types import SimpleNamespace

import bench


class Clock:
    """A lattice and CUDA events on a clock: a launch is one pass over the state at the
    peak rate and takes up to three steps."""

    def __init__(self, pass_ms):
        self.ms, self.pass_ms = 0.0, pass_ms
        self.cuda = SimpleNamespace(Event=lambda enable_timing: Event(self),
                                    synchronize=lambda: None)

    def step(self, n, kind, w=None):
        self.ms += -(-n // 3) * self.pass_ms

    def energy_spectrum(self, kmax):
        self.ms += self.pass_ms

    structure_functions = energy_spectrum


class Event:
    def __init__(self, clock):
        self.clock = clock

    def record(self, stream):
        self.ms = self.clock.ms

    def synchronize(self):
        pass

    def elapsed_time(self, end):
        return end.ms - self.ms


def fractions(d):
    for k, v in d.items():
        if isinstance(v, dict):
            yield from fractions(v)
        elif k.startswith("hbm"):
            yield k, v


def test_no_component_reads_above_the_bandwidth():
    n, peak = 4096, 6800.0
    clock = Clock(bench.BYTES_PER_NODE * n * n / (peak * 1e9) * 1e3)
    plain = bench._time_plain(clock, n * n, peak, 200, clock, None)
    assert plain["bgk_single_steps"]["hbm_frac"] == 1.0
    assert plain["smag_single_steps"]["hbm_gbs"] == peak
    assert plain["bgk"]["of_one_pass_per_step"] > 2.9
    diag = bench._time_diagnostics(clock, n, clock, None, peak)
    for k, v in [*fractions(plain), *fractions(diag)]:
        assert v <= (peak if k == "hbm_gbs" else 1.0), (k, v)
