"""The ends of steep tracks in the smoother's residuals (run on a GB300 with -m gpu).

After a fast fit the last clusters of tracks that end at |sin phi| > 0.9 go through
the square-root sequence, gathered from all over the batch, and all other clusters
through the combination of the tape's states.  Which one a track takes depends on
the track alone, and its ends are as close to 64 bits as the deterministic mode's,
which has the square-root sequence throughout."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2511_17018_gb300 import synth  # noqa: E402
from paper_2511_17018_gb300 import tpcfit as tf  # noqa: E402

ENDS = 16


@pytest.fixture(scope="module")
def steep():
    """A few hundred tracks that end steep or nearly so, of even and odd lengths, and |sin phi| of
    their last three clusters (64 bits)."""
    fr = synth.generate(30000, 64, drop_p=0.05)
    snp = np.abs(oracle.smooth_states(fr)["state"][:, 2])
    last = fr.offsets[1:].astype(np.int64) - 1
    three = np.stack([snp[np.maximum(last - k, 0)] for k in range(3)])
    pick = np.nonzero((fr.lengths() > 30) & np.isfinite(three).all(0) & (three.max(0) > 0.88))[0]
    return fr.subset(pick), three[:, pick]


def _repeat(dev, n):
    """The batch's tracks in turn, n of them, and each cluster's index in the batch."""
    m = dev["offsets"].numel() - 1
    idx = torch.arange(n, device="cuda") % m
    off = dev["offsets"].long()
    lens = (off[1:] - off[:-1])[idx]
    new = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=new[1:])
    owner = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
    src = off[idx][owner] + torch.arange(int(new[-1]), device="cuda") - new[owner]
    return dict(y=dev["y"][src], z=dev["z"][src], rowsec=dev["rowsec"][src], offsets=new.to(torch.int32),
                seeds=dev["seeds"][:, idx].contiguous()), src


def _smooth(fr, dev, det=False):
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=det)
    try:
        f.set_record(True)
        sm = f.smooth(dev, f.fit(dev))
        torch.cuda.synchronize()
        return sm
    finally:
        f.close()


@pytest.mark.parametrize("n", [2000, 38912, 38913, 50000])
def test_the_sequence_does_not_depend_on_the_batch(steep, n):
    # tracks that cross the line within their last three clusters, with an even and
    # an odd number of steps; every state on the tape up to 38,912 tracks, every
    # second one above
    fr, three = steep
    crossing = (three.min(0) < 0.9) & (three.max(0) > 0.9)
    even = fr.lengths() % 2 == 0
    assert (crossing & even).sum() >= 10 and (crossing & ~even).sum() >= 10
    dev = tf.frame_to_device(fr)
    alone = _smooth(fr, dev)
    big, src = _repeat(dev, n)
    got = _smooth(fr, big)
    for k in alone:
        assert torch.equal(got[k].view(torch.int32), alone[k][src].view(torch.int32)), k


def test_steep_ends_are_as_accurate_as_the_square_root_mode(steep):
    # fast mode's reciprocals and square roots are good to 2 units in the last place
    # instead of half a one: up to four times the rounding error
    fr, three = steep
    sel = np.nonzero(three[0] > 0.93)[0]
    assert len(sel) >= 50
    off = fr.offsets.astype(np.int64)
    ends = np.concatenate([np.arange(off[t + 1] - ENDS, off[t + 1]) for t in sel])
    ref = oracle.smooth(fr)
    dev = tf.frame_to_device(fr)
    err = []
    for det in (False, True):
        sm = {k: v.cpu().numpy().astype(np.float64) for k, v in _smooth(fr, dev, det).items()}
        e = {}
        for k in ("resid", "rcov", "chi2"):
            a, b = sm[k][ends], ref[k][ends]
            ok = np.isfinite(a) & np.isfinite(b)
            assert ok.mean() > 0.99, k
            e[k] = np.linalg.norm((a - b)[ok]) / np.linalg.norm(b[ok])
        err.append(e)
    print(err)
    for k in err[0]:
        assert err[0][k] <= 4 * err[1][k], (k, err)
