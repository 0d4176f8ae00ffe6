"""The voltage peaks that the reconstruction starts from, selected by FP32 sums of squares and decided in
FP64, against the oracle's (FP64 throughout): the first fit's direction, which moves by far more than the
tolerance if one station's sample differs. At scale 1, where the FP32 selection is in force, every station has
an earlier sample that ties with its peak in FP32 but not in FP64, a later one that FP32 puts above it and
FP64 below, and an exact tie (the lowest index wins). At the other scales the squares over- or underflow FP32 and
every sample goes to FP64."""
import numpy as np
import pytest

import oracle
from paper_1507_07733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


PEAK = np.float32([0.95667416, 0.76770145])


def _ulps(x, k):
    """x moved by k units in the last place (x > 0)."""
    return (x.view(np.int32) + np.int32(k)).view(np.float32)


TIE = np.float32([PEAK[0], _ulps(PEAK[1], -1)])                # the peak's FP32 sum, a smaller FP64 one
ABOVE = np.float32([_ulps(PEAK[0], -2), _ulps(PEAK[1], 2)])    # a larger FP32 sum, a smaller FP64 one


def _sum32(v):
    """fmaf(a, a, b * b) in FP32 (the FP64 sum has 29 bits more than the result: the second rounding is harmless
    unless it lands on a halfway case, which the assertions below would show)."""
    return np.float32(np.float64(v[0]) ** 2 + np.float64(np.float32(v[1] * v[1])))


def _sum64(v):
    return np.float64(v[0]) ** 2 + np.float64(v[1]) ** 2


def test_the_planted_samples_order_as_stated():
    assert _sum32(TIE) == _sum32(PEAK) < _sum32(ABOVE)
    assert max(_sum64(TIE), _sum64(ABOVE)) < _sum64(PEAK)


@pytest.mark.parametrize("n", [1024, 2048, 4096])
@pytest.mark.parametrize("scale", [1.0, 1e-21, 1e21, 1e-39])
def test_first_fit_follows_the_fp64_peaks(n, scale):
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pid = ctx.load_pattern(synth.make_pattern())
    ev = synth.make_event(30, n, synth.scan_directions(1, 1), seed_key=n)
    rng = np.random.default_rng(n)
    ev.traces[:] = rng.uniform(-0.5, 0.5, ev.traces.shape).astype(np.float32)
    at = n // 2 + rng.integers(0, 12, 30)
    for s, i in enumerate(at):
        ev.traces[s, :, i] = PEAK
        ev.traces[s, :, i - 1 - s] = TIE
        ev.traces[s, :, i + 40 + s] = ABOVE
        ev.traces[s, :, i + 80 + s] = -PEAK
    ev.traces *= np.float32(scale)
    idx, times = oracle.voltage_peaks(ev)
    if scale == 1.0:
        assert np.array_equal(idx, at)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ev.traces, ev.pos_m, ev.t_start_ns)]
    got = ctx.reconstruct(pid, *t, max_iter=1)["history"].cpu().numpy()[0]
    want = oracle.plane_fit(ev.pos_m, times)
    assert np.max(np.abs(got - want[:2])) <= 1e-9, (got, want)   # one sample (5 ns) of one station: 1e-5
    ctx.close()
