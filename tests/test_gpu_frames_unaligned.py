"""Frames that arrive during the launch in arrays of any alignment (run on a GB300
with -m gpu).

The staging copies clusters in windows of four that reach into the neighbouring
tracks, so next to a frame's boundary it reads words of the next frame that another
stream has yet to write; once that frame's flag is set, its own values have to be
seen.  Arrays that begin at one place within a window are copied in whole windows,
others cluster by cluster."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_17018_gb300 import synth  # noqa: E402
from paper_2511_17018_gb300 import tpcfit as tf  # noqa: E402
from paper_2511_17018_gb300.frames import FrameBatch, fit_frames  # noqa: E402

FRAMES, TRACKS = 150, 31


@pytest.mark.parametrize("lanes", [1, 4])
@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 1, 1), (3, 3, 3), (1, 2, 3), (0, 0, 1)])
def test_streamed_frames_at_any_alignment(shift, lanes):
    fr = synth.generate(FRAMES * TRACKS, 71, drop_p=0.05, cap_lengths=True)
    full = tf.frame_to_device(fr)
    base = torch.arange(0, FRAMES * TRACKS + 1, TRACKS, dtype=torch.int64, device="cuda")
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=True)
    try:
        f.set_config(lanes, 4, 24, True)
        ref = fit_frames(f, FrameBatch(full["y"], full["z"], full["rowsec"], full["offsets"], full["seeds"], base))
        ref = {k: v.clone() for k, v in ref.items()}
        assert f.status()[0] == tf.OK
        host, dev = {}, {}
        for k, s in zip(("y", "z", "rowsec"), shift):
            host[k] = full[k].cpu().pin_memory()
            # what is there before: no valid row, clusters far away
            dev[k] = torch.full((fr.n_hits + s,), -1 if k == "rowsec" else 1e3, dtype=full[k].dtype,
                                device="cuda")[s:]
        batch = FrameBatch(dev["y"], dev["z"], dev["rowsec"], full["offsets"], full["seeds"], base)
        flags = torch.zeros(FRAMES, dtype=torch.int32, device="cuda")
        one = torch.ones(1, dtype=torch.int32).pin_memory()
        out = tf.empty_outputs(batch.n_tracks)
        torch.cuda.synchronize()
        stream, copy = torch.cuda.Stream(), torch.cuda.Stream()
        with torch.cuda.stream(stream):
            fit_frames(f, batch, out, frame_ready=flags, wait_timeout_ns=2_000_000_000)
        with torch.cuda.stream(copy):
            for i in range(FRAMES):
                a, b = int(fr.offsets[i * TRACKS]), int(fr.offsets[(i + 1) * TRACKS])
                for k in ("y", "z", "rowsec"):
                    dev[k][a:b].copy_(host[k][a:b], non_blocking=True)
                flags[i:i + 1].copy_(one, non_blocking=True)
        torch.cuda.synchronize()
        assert f.status(stream)[0] == tf.OK
        for k in ("params", "cov", "chi2", "ndf"):
            assert torch.equal(out[k].view(torch.int32), ref[k].view(torch.int32)), k
    finally:
        f.close()
