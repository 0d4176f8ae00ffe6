"""The unfold kernel at the edges of its walk and of its inputs, against the oracle: one pair, a few pairs more than the
resident CTAs (152 x 2, 4 or 5), directions that end inside and at the end of a CTA's share, shares
of one pair and of several directions, and patterns from 2 to the most frequency nodes. Tolerances:
parity_util (1e-5 relative L2 per pair; measured 3e-7 to 5e-7). And stations with a NaN or an infinity."""
import numpy as np
import pytest

import oracle
from paper_1507_07733_gb300 import synth
from parity_util import check_event

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("n,s,d,n_freq", [
    (1024, 1, 1, 2), (1024, 5, 3, 193), (1024, 4, 2, 256), (1024, 23, 53, 51),
    (2048, 1, 1, 192), (2048, 3, 2, 256), (2048, 29, 21, 51),
    (1024, 1, 2300, 51), (2048, 57, 9, 51), (2048, 61, 11, 51),   # direction entries by CTAs of their own
    (4096, 1, 2, 256), (4096, 1, 306, 51), (4096, 61, 5, 98),
])
def test_edges_match_the_oracle(n, s, d, n_freq):
    from paper_1507_07733_gb300 import binding
    grid = dict(synth.PATTERN_GRID, n_zen=7, dzen_deg=15.0, n_az=24, daz_deg=15.0, n_freq=n_freq,
                df_hz=50e6 / (n_freq - 1))
    pat = synth.make_pattern(seed_key=n_freq, grid=grid)
    ev = synth.make_event(s, n, synth.random_directions(d, np.random.default_rng(n + s + d)), seed_key=2000 + s)
    ctx = binding.Context(0)
    pid = ctx.load_pattern(pat)
    out, struct = binding.alloc_outputs(d, s, n)
    args = (_dev(ev.traces), _dev(ev.pos_m), _dev(ev.t_start_ns), _dev(ev.dirs_rad))
    for _ in range(2):   # the second call reuses every workspace
        for v in out.values():
            v.fill_(-7)
        ctx.unfold(pid, *args, out=out, sync=True)
    gpu = {k: v.cpu().numpy() for k, v in out.items()}
    check_event(gpu, oracle.unfold_event(pat, ev), ev)
    ctx.close()


@pytest.mark.parametrize("n,s,d", [(1024, 9, 3), (2048, 124, 5), (4096, 7, 2)])
def test_a_station_of_nan_keeps_to_itself(n, s, d):
    """A NaN or an infinity in a station's trace makes its whole spectrum NaN: that station's traces are NaN, its
    peak is sample 0 with amplitude 0, and the other stations' outputs have the bits they have without it."""
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pid = ctx.load_pattern(synth.make_pattern())
    ev = synth.make_event(s, n, synth.random_directions(d, np.random.default_rng(n)), seed_key=2100 + s)
    bad = {2: np.nan, s - 1: np.inf}
    res = []
    for values in ({}, bad):
        for st, x in values.items():
            ev.traces[st, st % 2, n // 3] = x
        out = ctx.unfold(pid, _dev(ev.traces), _dev(ev.pos_m), _dev(ev.t_start_ns), _dev(ev.dirs_rad), sync=True)
        res.append({k: v.cpu().numpy() for k, v in out.items() if v is not None})
    good = [i for i in range(s) if i not in bad]
    for k in ("efield", "envelope", "peak_idx", "peak_amp", "peak_time_ns", "status"):
        assert np.array_equal(res[0][k][:, good], res[1][k][:, good]), k
    for st in bad:
        assert np.isnan(res[1]["efield"][:, st]).all() and np.isnan(res[1]["envelope"][:, st]).all()
        assert not res[1]["peak_idx"][:, st].any() and not res[1]["peak_amp"][:, st].any()
    ctx.close()
