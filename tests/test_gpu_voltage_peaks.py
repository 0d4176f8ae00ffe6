"""The voltage peaks that the reconstruction starts from, selected by FP32 sums of squares and decided in
FP64, against the oracle's (FP64 throughout): the first fit's direction, which moves by far more than the
tolerance if one station's sample differs. Samples that tie in FP32 but not in FP64, exact ties (the lowest
index wins), amplitudes whose squares over- or underflow FP32, and the lengths' remainders of a thread's stride."""
import numpy as np
import pytest

import oracle
from paper_1507_07733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1024, 2048, 4096])
@pytest.mark.parametrize("scale", [1.0, 1e-21, 1e21, 1e-39])
def test_first_fit_follows_the_fp64_peaks(n, scale):
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pid = ctx.load_pattern(synth.make_pattern())
    ev = synth.make_event(30, n, synth.scan_directions(1, 1), seed_key=n)
    rng = np.random.default_rng(n)
    ev.traces[:] = rng.uniform(-0.5, 0.5, ev.traces.shape).astype(np.float32)
    one, up = np.float32(1.0), np.nextafter(np.float32(1.0), np.float32(2.0))
    for s, i in enumerate(n // 2 + rng.integers(0, 12, 30)):
        ev.traces[s, :, i] = (up, up)               # the peak
        ev.traces[s, :, i - 1 - s] = (one, up)      # 1.2e-7 below it, earlier
        ev.traces[s, :, i + 40 + s] = (-up, up)     # the same, later
    ev.traces *= np.float32(scale)
    idx, times = oracle.voltage_peaks(ev)
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ev.traces, ev.pos_m, ev.t_start_ns)]
    got = ctx.reconstruct(pid, *t, max_iter=1)["history"].cpu().numpy()[0]
    want = oracle.plane_fit(ev.pos_m, times)
    assert np.max(np.abs(got - want[:2])) <= 1e-9, (got, want)   # one sample (5 ns) of one station: 1e-5
    ctx.close()
