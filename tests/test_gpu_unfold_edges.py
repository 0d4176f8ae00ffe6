"""The unfold kernel at the edges of its walk, against the oracle: one pair, a few pairs more than the
resident CTAs (152 x 2, 4 or 5), directions that end inside and at the end of a CTA's share, shares
of one pair and of several directions, and patterns from 2 to the most frequency nodes. Tolerances:
parity_util (1e-5 relative L2 per pair; measured 3e-7 to 5e-7)."""
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
