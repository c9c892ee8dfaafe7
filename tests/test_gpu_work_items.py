"""Work items of every size (run on a GB300 with -m gpu).

A small batch is cut into items of fewer than 32 tracks and spread over the SMs
with fewer warps per block; a track's result depends on that track alone, so it
must be the same bits in a batch of any size.  Sizes at the edges: one track,
one item per warp scheduler and one more, the one-block length ordering's
largest batch and one more, full items, one more than all resident warps hold."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from paper_2511_17018_gb300 import synth  # noqa: E402
from paper_2511_17018_gb300 import tpcfit as tf  # noqa: E402

POOL = 700
SIZES = (1, 2, 33, 607, 609, 1217, 16384, 16385, 19456, 19457, 38913, 116737)


@pytest.fixture(scope="module")
def pool():
    fr = synth.generate(POOL, 51, drop_p=0.05, cap_lengths=True)
    return fr, oracle.fit(fr, "f32")


def _repeat(fr, n):
    """The first n tracks of the pool repeated, on the device, and their pool indices."""
    idx = torch.arange(n, device="cuda") % fr.n_tracks
    d = tf.frame_to_device(fr)
    off = d["offsets"].to(torch.int64)
    lens = (off[1:] - off[:-1])[idx]
    new = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(lens, 0, out=new[1:])
    owner = torch.repeat_interleave(torch.arange(n, device="cuda"), lens)
    src = off[idx][owner] + torch.arange(int(new[-1]), device="cuda") - new[owner]
    return dict(y=d["y"][src], z=d["z"][src], rowsec=d["rowsec"][src], offsets=new.to(torch.int32),
                seeds=d["seeds"][:, idx].contiguous()), idx, src


def _bits(t):
    return t.contiguous().view(torch.int32)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("det", [False, True], ids=["fast", "det"])
def test_results_do_not_depend_on_the_batch_size(pool, n, det):
    fr, ref = pool
    dev, idx, src = _repeat(fr, n)
    full, fidx, fsrc = _repeat(fr, POOL)
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=det)
    try:
        f.set_record(True)
        out0 = f.fit(full)
        gm0 = torch.empty((full["y"].numel(), 2), device="cuda")
        _, gs0 = f.backward(full, out0, torch.ones(POOL, device="cuda"), gm0)
        sm0 = f.smooth(full, out0)
        out = f.fit(dev)
        gm = torch.empty((dev["y"].numel(), 2), device="cuda")
        _, gs = f.backward(dev, out, torch.ones(n, device="cuda"), gm)
        sm = f.smooth(dev, out)
        assert f.status()[0] == tf.OK
        for k in ("params", "cov", "chi2", "ndf"):
            assert torch.equal(_bits(out[k]), _bits(out0[k][..., idx])), k
            if det:
                want = torch.from_numpy(np.ascontiguousarray(ref[k])).cuda()[..., idx]
                assert torch.equal(_bits(out[k]), _bits(want)), k
        assert torch.equal(_bits(gs), _bits(gs0[:, idx]))
        assert torch.equal(_bits(gm), _bits(gm0[src]))
        for k in ("resid", "rcov", "chi2"):
            assert torch.equal(_bits(sm[k]), _bits(sm0[k][src])), k
    finally:
        f.close()
