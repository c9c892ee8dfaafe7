"""Work items of every size (run on a GB300 with -m gpu).

A small batch is cut into items of fewer than 32 tracks and spread over the SMs
with fewer warps per block; a track's result depends on that track alone, so it
must be the same bits in a batch of any size.  Sizes at the edges: one track,
one item per warp scheduler and one more, the one-block length ordering's
largest batch and one more, full items, one more than all resident warps hold.
A recorded fit keeps every state of a small batch and every second one of a
large one, and an item that finds no room for its states leaves checkpoints: the
gradients are the same either way."""
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


@pytest.mark.parametrize("mode", ["fast", "det", "material"])
def test_items_without_room_on_the_tape_leave_checkpoints(mode):
    # Tracks of three clusters a row (up to 456) in a batch that is not sorted by
    # length: room for 152 steps an item is reserved, so most items of two tracks
    # find none.  The same tracks, 600 of them in items of one track that all find
    # room, are the reference: bit for bit in the deterministic mode, whose reverse
    # has one operation sequence; in the fast modes both kernels compute the same
    # formulas on the same states, so they differ by the rounding of the reverse at
    # most (1e-5 in norm).
    fr = synth.generate(1000, 52)
    off = fr.offsets.astype(np.int64)
    three = np.repeat(np.arange(fr.n_hits), 3)
    dev = tf.frame_to_device(fr)
    pick = torch.from_numpy(three).cuda()
    dev = dict(y=dev["y"][pick], z=dev["z"][pick], rowsec=dev["rowsec"][pick],
               offsets=torch.from_numpy((3 * off).astype(np.int32)).cuda(), seeds=dev["seeds"])
    n, h = 600, int(3 * off[600])
    part = dict(y=dev["y"][:h].contiguous(), z=dev["z"][:h].contiguous(), rowsec=dev["rowsec"][:h].contiguous(),
                offsets=dev["offsets"][:n + 1].contiguous(), seeds=dev["seeds"][:, :n].contiguous())
    got = []
    for d, srt in ((part, True), (dev, False)):
        f = tf.Fitter(fr.geometry, fr.bz, deterministic=mode == "det", sort_by_length=srt)
        try:
            f.set_material(synth.TPC_GAS if mode == "material" else None)
            f.set_record(True)
            out = f.fit(d)
            gm = torch.empty((d["y"].numel(), 2), device="cuda")
            _, gs = f.backward(d, out, torch.ones(d["offsets"].numel() - 1, device="cuda"), gm)
            sm = f.smooth(d, out)["chi2"]
            assert f.status()[0] == tf.OK
            assert int((out["ndf"] > 400).sum()) > 300
            got.append((gm[:h].clone(), gs[:, :n].clone(), sm[:h].clone()))
        finally:
            f.close()
    for a, b in zip(*got):
        if mode == "det":
            assert torch.equal(_bits(a), _bits(b))
        else:
            a, b = a.double(), b.double()
            assert torch.equal(torch.isnan(a), torch.isnan(b))
            assert float((a - b).nan_to_num().norm()) <= 1e-5 * float(a.nan_to_num().norm())


@pytest.mark.parametrize("shift", [1, 2, 3, 4])
@pytest.mark.parametrize("det", [False, True], ids=["fast", "det"])
def test_clusters_at_any_alignment(pool, shift, det):
    # the clusters of 700 tracks begin `shift` elements into their arrays, which end
    # with the last cluster: windows of 4 are whole, cut off at the end, or (not a
    # multiple of 4 elements) not aligned at all; in the middle of the arrays they
    # reach into the neighbouring tracks
    fr, _ = pool
    full, _, _ = _repeat(fr, POOL)

    def moved(t):
        big = torch.zeros(t.numel() + shift, dtype=t.dtype, device="cuda")
        big[shift:] = t
        return big[shift:]

    dev = dict(full, y=moved(full["y"]), z=moved(full["z"]), rowsec=moved(full["rowsec"]))
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=det)
    try:
        a, b = f.fit(full), f.fit(dev)
        assert f.status()[0] == tf.OK
        for k in ("params", "cov", "chi2", "ndf"):
            assert torch.equal(_bits(a[k]), _bits(b[k])), k
    finally:
        f.close()


def test_the_recording_outlives_other_settings(pool):
    # the adjoint follows the recorded fit's order of the tracks, whatever the sort
    # switch and the reserved size are by then
    fr, _ = pool
    dev, _, _ = _repeat(fr, POOL)
    g = torch.ones(POOL, device="cuda")
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=True)
    try:
        f.set_record(True)
        out = f.fit(dev)
        ga, gs = f.backward(dev, out, g)
        sm = f.smooth(dev, out)["chi2"]
        f.set_config(sort_by_length=False)
        tf.tpcfit_reserve(f.h, 3_000_000)
        ga2, gs2 = f.backward(dev, out, g)
        sm2 = f.smooth(dev, out)["chi2"]
        assert torch.equal(_bits(ga), _bits(ga2)) and torch.equal(_bits(gs), _bits(gs2))
        assert torch.equal(_bits(sm), _bits(sm2))
    finally:
        f.close()
