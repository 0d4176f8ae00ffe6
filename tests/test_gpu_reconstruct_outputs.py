"""The reconstruction with each set of outputs: without SNRs the unfold kernel's last CTA makes an iteration's
fit, with them a kernel of its own does. The fit takes whole-sample times and no weights, so both give the same
bits. And fits that leave the sky (nx^2 + ny^2 > 1), which end on the horizon, against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1507_07733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _reconstruct(binding, ctx, pid, args, max_iter, **modes):
    s, _, n = args[0].shape
    last, _ = binding.alloc_outputs(1, s, n, **modes)
    f64 = dict(dtype=torch.float64, device="cuda")
    res = dict(direction=torch.empty(2, **f64), t0_ns=torch.empty(1, **f64), chi2=torch.empty(1, **f64),
               iterations=torch.empty(1, dtype=torch.int32, device="cuda"), history=torch.empty((max_iter + 1, 2), **f64))
    ev = binding.make_event(pid, *args, torch.empty((1, 2), **f64))
    out = binding.ar_recon_out(*(res[k].data_ptr() for k in ("direction", "t0_ns", "chi2", "iterations", "history")),
                               binding.outputs_struct(last))
    binding.ar_reconstruct(ctx.h, ev, max_iter, 1e-6, out, torch.cuda.current_stream().cuda_stream)
    ctx.sync()
    return {k: v.cpu().numpy() for k, v in res.items()}, {k: v for k, v in last.items() if v is not None}


@pytest.mark.parametrize("s,n,key", [(20, 1024, 72), (124, 2048, 74), (60, 4096, 73)])
def test_every_set_of_outputs_gives_the_same_loop(s, n, key):
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pid = ctx.load_pattern(synth.make_pattern())
    ev = synth.make_event(s, n, synth.scan_directions(1, 1), seed_key=key)
    args = [_dev(a) for a in (ev.traces, ev.pos_m, ev.t_start_ns)]
    plain, plain_last = _reconstruct(binding, ctx, pid, args, 8)
    it = int(plain["iterations"][0])
    assert 0 < it < 8   # converged: launches after it return at once
    for modes in (dict(snr=True), dict(fine=True), dict(snr=True, fine=True), dict(snr=True, traces=False)):
        res, last = _reconstruct(binding, ctx, pid, args, 8, **modes)
        for k in plain:
            assert np.array_equal(plain[k], res[k], equal_nan=True), (modes, k)
        out, _ = binding.alloc_outputs(1, s, n, **modes)   # the last unfold again, by itself
        ctx.unfold(pid, *args, _dev(plain["history"][it - 1:it]), out=out, sync=True)
        for k in ("peak_idx", "peak_amp", "peak_time_ns", "status", "peak_time_fine_ns", "snr", "efield", "envelope"):
            if last.get(k) is not None:
                assert torch.equal(last[k], out[k]), (modes, k)
    ctx.close()


@pytest.mark.parametrize("s,n,max_iter", [(30, 1024, 0), (30, 2048, 2), (124, 4096, 3)])
def test_a_fit_beyond_the_horizon_ends_on_it(s, n, max_iter):
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pat = synth.make_pattern()
    pid = ctx.load_pattern(pat)
    ev = synth.make_event(s, n, synth.scan_directions(1, 1), seed_key=s)
    ev.t_start_ns[:] -= ev.pos_m[:, :2] @ np.array([1.7, -2.3]) / 0.299792458   # a wave slower than light
    r = oracle.reconstruct(pat, ev, max_iter=max_iter, tol_rad=1e-6)
    got, _ = _reconstruct(binding, ctx, pid, [_dev(a) for a in (ev.traces, ev.pos_m, ev.t_start_ns)], max_iter)
    assert got["iterations"][0] == r["iterations"]
    assert abs(r["zenith"] - np.pi / 2) < 1e-12
    assert np.allclose(got["direction"], (r["zenith"], r["azimuth"]), rtol=0, atol=1e-9)
    assert np.allclose(got["history"], r["history"], rtol=0, atol=1e-9, equal_nan=True)
    for k in ("t0_ns", "chi2"):
        assert abs(got[k][0] - r[k]) <= 1e-9 * max(1.0, abs(r[k]))
    ctx.close()
