"""What a recording holds, and for which tracks and clusters the adjoint and the
smoother answer (run on a GB300 with -m gpu)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_17018_gb300 import synth  # noqa: E402
from paper_2511_17018_gb300 import tpcfit as tf  # noqa: E402

# name: deterministic, lanes per track, factor of the fast fit and reverse, material
KINDS = {"fast": (False, 1, 1, False), "det": (True, 1, 1, False), "material": (False, 1, 1, True),
         "fast_checkpoints": (False, 1, 0, False), "det_checkpoints": (True, 8, 1, False)}


def _fitter(fr, kind):
    det, lanes, form, material = KINDS[kind]
    f = tf.Fitter(fr.geometry, fr.bz, deterministic=det)
    f.set_config(lanes, 4, 24, True)
    f.set_fit_form(form)
    f.set_backward_form(form)
    f.set_material(synth.TPC_GAS if material else None)
    f.set_record(True)
    return f


def _bits(t):
    return t.contiguous().view(torch.int32)


class Guarded:
    """A tensor of n elements in the middle of a larger one that has to stay as it is."""

    def __init__(self, *shape, margin=1024):
        n = int(np.prod(shape))
        self.big = torch.full((n + 2 * margin,), 7.0, device="cuda")
        self.t = self.big[margin:margin + n].view(*shape)
        self.margin = margin

    def intact(self):
        m = self.margin
        return bool((self.big[:m] == 7.0).all()) and bool((self.big[-m:] == 7.0).all())


def _follow(f, dev, ndf):
    """Adjoint, residuals and states of the recorded fit, into guarded outputs."""
    n = dev["offsets"].numel() - 1
    H = dev["y"].numel()
    o = dict(ga=Guarded(36 * 152 * 2), gs=Guarded(5, n), gm=Guarded(H, 2), resid=Guarded(H, 2), rcov=Guarded(H, 3),
             chi2=Guarded(H), state=Guarded(H, 5), state_cov=Guarded(H, 15))
    args = (f.h, dev["y"], dev["z"], dev["rowsec"], dev["offsets"], ndf)
    tf.tpcfit_fit_backward(*args, torch.ones(n, device="cuda"), o["ga"].t, o["gs"].t, o["gm"].t)
    tf.tpcfit_smooth(*args, o["resid"].t, o["rcov"].t, o["chi2"].t)
    tf.tpcfit_smooth_states(*args, o["state"].t, o["state_cov"].t)
    torch.cuda.synchronize()
    for k, v in o.items():
        assert v.intact(), k
    return {k: v.t for k, v in o.items()}


@pytest.mark.parametrize("kind", KINDS)
def test_the_recording_decides_which_tracks_were_fitted(kind):
    # another fit's ndf calls tracks fitted that the recorded fit could not start:
    # the recording holds nothing of them, so they count as not fitted
    fr = synth.generate(300, 61)
    dev = tf.frame_to_device(fr)
    bad = torch.arange(0, 300, 7, device="cuda")
    unusable = dict(dev, seeds=dev["seeds"].clone())
    unusable["seeds"][2, bad] = 0.9995
    f = _fitter(fr, kind)
    try:
        ndf_other = f.fit(dev)["ndf"].clone()
        out = f.fit(unusable)
        assert bool((ndf_other[bad] > 0).all()) and bool((out["ndf"][bad] == -1).all())
        got = _follow(f, unusable, torch.where(out["ndf"] > 0, out["ndf"], ndf_other))
        want = _follow(f, unusable, out["ndf"])
        assert bool((got["gs"][:, bad] == 0).all())
        for k in want:
            if k == "ga" and not KINDS[kind][0]:  # atomics: the order of the additions is free
                assert float((got[k] - want[k]).norm()) <= 1e-5 * float(want[k].norm())
            else:
                assert torch.equal(_bits(got[k]), _bits(want[k])), k
    finally:
        f.close()


@pytest.mark.parametrize("where", ["last", "middle"])
@pytest.mark.parametrize("kind", KINDS)
def test_offsets_beyond_the_arrays_touch_nothing_outside(kind, where):
    # an offset beyond the cluster arrays: the fit flags the tracks it bounds, the
    # adjoint and the smoother leave everything outside the arrays alone and give
    # the other tracks what they get with good offsets
    fr = synth.generate(300, 62)
    dev = tf.frame_to_device(fr)
    H = fr.n_hits
    at = 300 if where == "last" else 120
    bad = [299] if where == "last" else [119, 120]
    broken = dict(dev, offsets=dev["offsets"].clone())
    for k in ("y", "z", "rowsec"):  # the arrays as views of larger ones
        big = torch.zeros(H + 2048, dtype=dev[k].dtype, device="cuda")
        big[1024:1024 + H] = dev[k]
        broken[k] = big[1024:1024 + H]
    broken["offsets"][at] = H + 5
    keep = torch.ones(300, dtype=torch.bool, device="cuda")
    keep[bad] = False
    owner = torch.repeat_interleave(torch.arange(300, device="cuda"), (dev["offsets"][1:] - dev["offsets"][:-1]).long())
    mine = keep[owner]
    f = _fitter(fr, kind)
    try:
        want = _follow(f, dev, f.fit(dev)["ndf"])
        assert f.status()[0] == tf.OK
        out = f.fit(broken)
        assert bool((out["ndf"][bad] == -2).all())
        got = _follow(f, broken, out["ndf"])
        st, code, trk = f.status()
        assert st == tf.EDEVICE and code == 1 and trk in bad
        assert torch.equal(_bits(got["gs"][:, keep]), _bits(want["gs"][:, keep]))
        assert bool((got["gs"][:, bad] == 0).all()) and bool((got["gm"][~mine] == 0).all())
        for k in ("gm", "resid", "rcov", "chi2", "state", "state_cov"):
            assert torch.equal(_bits(got[k][mine]), _bits(want[k][mine])), k
        if where == "last":  # in order, but for the arrays' end
            for k in ("resid", "rcov", "chi2", "state", "state_cov"):
                assert bool(torch.isnan(got[k][~mine]).all()), k
    finally:
        f.close()


def _ends_early(n, seed, step=20):
    """Tracks of which every third has cluster `step` in the sector opposite, where no
    step leads: its outward pass ends there."""
    fr = synth.generate(n, seed)
    fr.rowsec = fr.rowsec.copy()
    off = fr.offsets.astype(np.int64)
    early = np.array([t for t in range(0, n, 3) if off[t + 1] - off[t] > step + 5])
    for t in early:
        h = off[t] + step
        row, sec = int(fr.rowsec[h]) >> 6, int(fr.rowsec[h]) & 63
        fr.rowsec[h] = np.uint16((row << 6) | (sec // 18 * 18 + (sec + 9) % 18))
    return fr, early, step


@pytest.mark.parametrize("reduction", [0, 1])
@pytest.mark.parametrize("kind", KINDS)
def test_clusters_that_no_step_reached_have_no_gradient(kind, reduction):
    # clusters after the end of an outward pass, and clusters of no track at all:
    # their gradients are zero and no alignment gradient holds what another call,
    # or nobody, left in their place
    fr, early, step = _ends_early(300, 63)
    whole = tf.frame_to_device(fr)
    dev = dict(whole, offsets=whole["offsets"][1:-1].contiguous(), seeds=whole["seeds"][:, 1:-1].contiguous())
    off = fr.offsets[1:-1].astype(np.int64)
    n = 298
    end = off[1:].copy()
    inner = early[(early > 0) & (early < 299)]
    end[inner - 1] = off[inner - 1] + step
    reached = np.zeros(fr.n_hits, bool)
    for t in range(n):
        reached[off[t]:end[t]] = True
    reached_dev = torch.from_numpy(reached).cuda()
    g = torch.ones(n, device="cuda")
    ga = []
    for used_before in (True, False):
        f = _fitter(fr, kind)
        try:
            f.set_det_reduction(reduction)
            if used_before:  # the handle's scratch holds large gradients of all clusters
                straight = tf.frame_to_device(synth.generate(300, 63))
                out = f.fit(straight)
                f.backward(straight, out, torch.full((300,), 1e4, device="cuda"))
            out = f.fit(dev)
            assert f.status()[0] == tf.OK
            assert bool((out["ndf"][torch.from_numpy(inner - 1).cuda()] == 2 * step - 5).all())
            ga.append(f.backward(dev, out, g)[0].reshape(-1, 2).clone())
            gm = torch.full((fr.n_hits, 2), 9.0, device="cuda")
            f.backward(dev, out, g, gm)
            assert bool((gm[~reached_dev] == 0).all()) and bool((gm[reached_dev] != 9.0).all())
        finally:
            f.close()
        # each alignment gradient is minus the sum of its clusters' (FP32 sums of a
        # few terms: 1e-5 in norm)
        key = torch.from_numpy((fr.rowsec.astype(np.int64) & 63) * 152 + (fr.rowsec.astype(np.int64) >> 6)).cuda()
        want = torch.zeros((36 * 152, 2), dtype=torch.float64, device="cuda").index_add_(0, key, -gm.double())
        assert float((ga[-1].double() - want).norm()) <= 1e-5 * float(want.norm())
    if KINDS[kind][0]:
        assert torch.equal(_bits(ga[0]), _bits(ga[1]))


def test_a_captured_fit_and_adjoint_outlive_larger_calls():
    # the graph's tape and scratch stay in place while the handle goes on to fits
    # that need more of both
    fr = synth.generate(3000, 65, drop_p=0.05, cap_lengths=True)
    dev = tf.frame_to_device(fr)
    large = tf.frame_to_device(synth.generate(20000, 66))
    g, g_large = torch.ones(3000, device="cuda"), torch.ones(20000, device="cuda")
    f = tf.Fitter(fr.geometry, fr.bz)
    try:
        f.set_record(True)
        out = tf.empty_outputs(3000)
        ga, gs = f.backward(dev, f.fit(dev, out), g)
        want = {k: out[k].clone() for k in out}
        ga0, gs0 = ga.clone(), gs.clone()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            ga, gs = f.backward(dev, f.fit(dev, out), g)
        for det in (True, False):
            f.set_mode(det)
            o = f.fit(large)
            f.backward(large, o, g_large)
            f.smooth(large, o)
        junk = [torch.full((1 << 26,), 3.0, device="cuda") for _ in range(8)]  # takes what was given back
        torch.cuda.synchronize()
        for t in (*out.values(), gs):
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for k in out:
            assert torch.equal(_bits(out[k]), _bits(want[k])), k
        assert torch.equal(_bits(gs), _bits(gs0))
        assert float((ga - ga0).norm()) <= 1e-5 * float(ga0.norm())
        assert all(bool((t == 3.0).all()) for t in junk)
        del graph
    finally:
        f.close()
