"""Calls queued behind one another without a synchronisation, the inputs rewritten in place by device
kernels between them: the same bits as synchronised calls. The kernels of a call start before the ones ahead
of them have ended, and some read directions, traces and tables before any wait of their own."""
import numpy as np
import pytest

from paper_1507_07733_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

RATES = (200e6, 220e6, 240e6)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _bits(out):
    return {k: v.clone() for k, v in out.items() if v is not None}


def _same(a, b):
    return all(torch.equal(a[k].contiguous().view(torch.uint8), b[k].contiguous().view(torch.uint8)) for k in a)


@pytest.mark.parametrize("entry", ["unfold", "noalloc", "tc", "reconstruct"])
@pytest.mark.parametrize("s,n,d", [(7, 2048, 3), (40, 1024, 30), (124, 4096, 2), (60, 4096, 9)])
def test_rewritten_inputs_are_read_as_of_the_call(entry, s, n, d):
    from paper_1507_07733_gb300 import binding
    ctx = binding.Context(0)
    pats = [synth.make_pattern(seed_key=k) for k in range(3)]
    pid = ctx.load_pattern(pats[0])
    p = pats[0]
    desc = dict(n_zen=p.n_zen, zen0_rad=p.zen0_rad, dzen_rad=p.dzen_rad, n_az=p.n_az, az0_rad=p.az0_rad,
                daz_rad=p.daz_rad, n_freq=p.n_freq, f0_hz=p.f0_hz, df_hz=p.df_hz)
    tables = [_dev(q.table.view(np.float32)) for q in pats]
    evs = [synth.make_event(s, n, synth.random_directions(d, np.random.default_rng(k)), seed_key=60 + k,
                            fs_hz=RATES[k]) for k in range(3)]
    src = [[_dev(a) for a in (e.traces, e.pos_m, e.t_start_ns, e.dirs_rad)] + [t] for e, t in zip(evs, tables)]
    buf = [x.clone() for x in src[0]]
    out, struct = binding.alloc_outputs(d, s, n)
    stream = torch.cuda.current_stream().cuda_stream

    def call(k):   # the result's tensors, the sample rate (and with it the tables) of event k
        for b, x in zip(buf, src[k]):
            torch.mul(x, 1.0, out=b)
        if entry == "reconstruct":
            r = ctx.reconstruct(pid, *buf[:3], fs_hz=RATES[k], sync=False)
            return _bits({**{q: v for q, v in r.items() if q != "last"}, **r["last"]})
        ev = binding.make_event(pid, *buf[:4], RATES[k])
        if entry == "unfold":
            binding.ar_unfold(ctx.h, ev, struct, stream)
        elif entry == "tc":
            binding.ar_unfold_tc(ctx.h, ev, struct, 6, stream)
        else:
            binding.ar_unfold_noalloc(desc, buf[4].data_ptr(), ev, struct, stream)
        return _bits(out)

    ref = []
    for k in range(3):
        torch.cuda.synchronize()
        ref.append(call(k))
        torch.cuda.synchronize()
    got = [(i % 3, call(i % 3)) for i in range(30)]
    ctx.sync()
    assert not _same(ref[0], ref[1])
    assert [i for i, (k, g) in enumerate(got) if not _same(g, ref[k])] == []
    ctx.close()
