"""Clusters in arrays that begin anywhere within a window of four (run on a GB300 with
-m gpu).

The fit stages aligned windows: arrays that all begin at the same place within one
share them, others are copied in smaller pieces (full batches) or cluster by cluster.
Every way has to give the bits of aligned arrays, to the first and last cluster."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_17018_gb300 import synth  # noqa: E402
from paper_2511_17018_gb300 import tpcfit as tf  # noqa: E402
from paper_2511_17018_gb300.frames import FrameBatch, fit_frames  # noqa: E402

POOL = 700
# where y, z and rowsec begin within their windows
PLACES = [(1, 1, 1), (2, 2, 2), (3, 3, 3), (1, 2, 3), (0, 2, 0), (0, 1, 0), (0, 0, 2), (3, 0, 1)]


def _batch(fr, n):
    d = tf.frame_to_device(fr)
    idx = torch.arange(n, device="cuda") % fr.n_tracks
    off = d["offsets"].long()
    lens = (off[1:] - off[:-1])[idx]
    new = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=new[1:])
    owner = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
    src = off[idx][owner] + torch.arange(int(new[-1]), device="cuda") - new[owner]
    return dict(y=d["y"][src], z=d["z"][src], rowsec=d["rowsec"][src], offsets=new.to(torch.int32),
                seeds=d["seeds"][:, idx].contiguous())


def _moved(t, k):
    big = torch.zeros(t.numel() + k, dtype=t.dtype, device="cuda")
    big[k:] = t
    return big[k:]


# one track, ragged batches, and the first size at which a batch fills blocks of 24 warps
@pytest.mark.parametrize("n", [1, 5, 700, 80000])
@pytest.mark.parametrize("mode", ["fast", "det", "material"])
def test_arrays_that_begin_anywhere_give_the_same_bits(n, mode):
    fr = synth.generate(POOL, 81, drop_p=0.05, cap_lengths=True)
    dev = _batch(fr, n)
    base = torch.tensor([0, n // 2, n], dtype=torch.int64, device="cuda")
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=mode == "det")
    f.set_material(synth.TPC_GAS if mode == "material" else None)

    def results(d):
        out = [f.fit(d)]
        out.append(fit_frames(f, FrameBatch(d["y"], d["z"], d["rowsec"], d["offsets"], d["seeds"], base)))
        f.set_record(True)
        rec = f.fit(d)
        _, gs = f.backward(d, rec, torch.ones(n, device="cuda"))
        f.set_record(False)
        assert f.status()[0] == tf.OK
        return [t for o in out for t in o.values()] + list(rec.values()) + [gs]

    try:
        want = results(dev)
        for places in PLACES:
            d = dict(dev, **{k: _moved(dev[k], s) for k, s in zip(("y", "z", "rowsec"), places)})
            for a, b in zip(results(d), want):
                assert torch.equal(a.contiguous().view(torch.int32), b.contiguous().view(torch.int32)), places
    finally:
        f.close()
