"""The tensor-core variant's two post-passes, in the inverse GEMM's epilogue (events of more than 152 tiles
of 128 x 128) and in a kernel of its own (asked for by an output that needs a pair's whole
envelope): the same operations in the same order, so the same bits. Pair counts at the least that takes the
epilogue, ends inside a tile's 128 rows, two chunks of pairs of which the second is too small for it; one
station of NaN and one of zeros; peaks without traces."""
import numpy as np
import pytest

from paper_1507_07733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,s,d,terms,traces", [
    (4096, 17, 9, 6, True), (4096, 17, 9, 3, False), (4096, 43, 29, 3, True),
    (2048, 61, 5, 6, True), (2048, 31, 23, 3, False), (1024, 29, 21, 6, True), (1024, 101, 13, 3, True),
    (4096, 124, 67, 6, False),
])
def test_epilogue_equals_the_post_pass(n, s, d, terms, traces):
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pid = ctx.load_pattern(synth.make_pattern())
    ev = synth.make_event(s, n, synth.random_directions(d, np.random.default_rng(n + s)), seed_key=3000 + s)
    ev.traces[3, 0, 17] = np.nan
    ev.traces[5] = 0.0
    args = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ev.traces, ev.pos_m, ev.t_start_ns, ev.dirs_rad)]
    res = []
    for snr in (False, True):
        out, _ = binding.alloc_outputs(d, s, n, traces=traces, snr=snr)
        for v in out.values():
            if v is not None:
                v.fill_(-7)
        ctx.unfold_tc(pid, *args, split_terms=terms, out=out, sync=True)
        res.append(out)
    for k in ("efield", "envelope", "peak_idx", "peak_amp", "peak_time_ns", "status"):
        a, b = res[0][k], res[1][k]
        if a is None:
            continue
        a, b = a.view(torch.uint8), b.view(torch.uint8)
        nan = torch.isnan(res[0][k]) & torch.isnan(res[1][k]) if k in ("efield", "envelope") else None
        if nan is not None:
            a, b = res[0][k].masked_fill(nan, 0).view(torch.uint8), res[1][k].masked_fill(nan, 0).view(torch.uint8)
        assert torch.equal(a, b), k
    ctx.close()
