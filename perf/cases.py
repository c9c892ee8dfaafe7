"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call, or one chain of calls, through the Python binding of the C ABI: the plain fit, the fit of many
time frames in one launch, the fit with checkpoints followed by its adjoint (device buffers, or host buffers), the
two-filter smoother, the smoothed states, and the outlier rejection.  `prepare` simulates the tracks on the GPU with
the distributions of `synth` (exact helices through the pad rows, dropped and smeared clusters, three-point seeds);
`exact` is the same filter written out in plain torch at 64 bits (covariance form), its gradient by torch's
automatic differentiation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_17018_gb300 import synth
from paper_2511_17018_gb300 import tpcfit as tf
from paper_2511_17018_gb300.frames import FrameBatch, fit_frames

DEV = "cuda"
F64 = torch.float64
ROWS = synth.N_ROWS
#: clusters per track: every row crossed, or 5% of them dropped and at most U{10..152} kept
MEAN_HITS = {"natural": 151.7, "capped": 80.6}
#: the field map and the drift gas of the runs that correct for them
FIELD = synth.FieldMap(0.3, -0.2)
GAS = synth.TPC_GAS


def listed():
    return [
        # one small frame, as a monitoring task or a test beam run fits it: latency and launches count
        dict(name="fit_1k", kind="fit", tracks=1000, lengths="natural"),
        # a slice of a frame in the non-uniform field, as a calibration pass fits it; ragged sizes
        dict(name="fit_20k_field", kind="fit", tracks=20011, lengths="capped", field=True),
        # a whole time frame: the reconstruction itself
        dict(name="fit_400k", kind="fit", tracks=400_000, lengths="capped"),
        # uneven time frames in one launch, each with alignment constants of its own
        dict(name="frames_40", kind="frames", frames=40, lo=1000, hi=60_000),
        # gradient of a small sample: an alignment or calibration loop on few tracks
        dict(name="adjoint_1k", kind="adjoint", tracks=1000, lengths="natural"),
        # gradient of a sample with alignment offsets, with the gradient of every cluster
        dict(name="adjoint_100k", kind="adjoint", tracks=100_000, lengths="capped", align=True, meas=True),
        # a whole time frame from pinned host buffers and its gradients back: a stream of frames being aligned
        dict(name="adjoint_host_400k", kind="adjoint_host", tracks=400_000, lengths="capped"),
        # the reproducible mode, as validation against a CPU runs it
        dict(name="adjoint_det_50k", kind="adjoint", tracks=50_000, lengths="capped", det=True, align=True),
        # energy loss, multiple scattering and the field map followed
        dict(name="adjoint_physics_20k", kind="adjoint", tracks=20_000, lengths="capped", material=True, field=True),
        # quality control: leave-one-out residuals of every cluster
        dict(name="smooth_100k", kind="smooth", tracks=100_000, lengths="capped"),
        # track state and covariance at every cluster, as dE/dx and distortion maps take them
        dict(name="states_30k", kind="states", tracks=30_011, lengths="capped"),
        # the clusters above a chi2 cut dropped before a refit
        dict(name="reject_200k", kind="reject", tracks=200_000, lengths="capped"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["fit", "fit", "frames", "adjoint", "adjoint", "adjoint_host", "smooth", "states", "reject"])
    lengths = rng.choice(["natural", "capped", "capped"])
    if kind == "fit":
        return dict(kind=kind, tracks=size(50, 400_000), lengths=lengths, det=rng.random() < 0.25,
                    field=rng.random() < 0.25, align=rng.random() < 0.5)
    if kind == "frames":
        return dict(kind=kind, frames=rng.randint(2, 40), lo=rng.randint(200, 2000), hi=size(5000, 60_000))
    if kind == "adjoint":
        physics = rng.choice(["plain", "plain", "det", "field", "material"])
        hi = {"plain": 200_000, "det": 50_000, "field": 100_000, "material": 30_000}[physics]
        return dict(kind=kind, tracks=size(100, hi), lengths=lengths, det=physics == "det",
                    field=physics in ("field", "material"), material=physics == "material",
                    align=rng.random() < 0.5, meas=rng.random() < 0.5)
    if kind == "adjoint_host":
        return dict(kind=kind, tracks=size(5000, 400_000), lengths="capped")
    if kind == "smooth":
        return dict(kind=kind, tracks=size(1000, 100_000), lengths=lengths)
    if kind == "states":
        return dict(kind=kind, tracks=size(1000, 40_000), lengths=lengths)
    return dict(kind=kind, tracks=size(1000, 200_000), lengths=lengths)


# ---------------------------------------------------------------- inputs
def _wrap(a):
    return torch.remainder(a + math.pi, 2.0 * math.pi) - math.pi


def _simulate(n, gen, lengths, d_true):
    """n candidate tracks through the pad rows (the recipe of synth.simulate, vectorised over tracks):
    y, z, sector of every row and whether a cluster is kept there, all [rows, n]."""
    rows_x = synth.default_geometry().row_x
    width = math.radians(20.0)
    half_tan = math.tan(0.5 * width)

    def uniform(lo, hi):
        return lo + (hi - lo) * torch.rand(n, generator=gen, device=DEV, dtype=F64)

    q = torch.where(uniform(0, 1) < 0.5, 1.0, -1.0).to(F64)
    k = synth.KAPPA_PER_TESLA * 0.5 * q * torch.exp(-uniform(math.log(0.2), math.log(10.0)))
    tanl = torch.sinh(uniform(-0.9, 0.9))
    phi0 = uniform(0.0, 2.0 * math.pi)
    z0 = 5.0 * torch.randn(n, generator=gen, device=DEV, dtype=F64)
    drop = torch.rand((ROWS, n), generator=gen, device=DEV) < (0.05 if lengths == "capped" else 0.0)
    xc, yc = -torch.sin(phi0) / k, torch.cos(phi0) / k
    hy = torch.zeros((ROWS, n), device=DEV, dtype=F64)
    hz = torch.zeros_like(hy)
    hs = torch.zeros((ROWS, n), device=DEV, dtype=torch.int64)
    keep = torch.zeros((ROWS, n), device=DEV, dtype=torch.bool)
    alive = torch.ones(n, device=DEV, dtype=torch.bool)
    l_prev = torch.zeros(n, device=DEV, dtype=F64)
    cand = torch.floor(phi0 / width).to(torch.int64) % 18

    def cross(sec, xr):
        a = (sec + 0.5) * width
        ca, sa = torch.cos(a), torch.sin(a)
        u = k * (xr - (xc * ca + yc * sa))
        uu = u.clamp(-0.999999, 0.999999)
        y = (-xc * sa + yc * ca) - torch.sqrt(1.0 - uu * uu) / k
        return u, y, _wrap(a + torch.asin(uu) - phi0) / k

    for r in range(ROWS):
        xr = float(rows_x[r])
        u, y, l = cross(cand, xr)
        out = y.abs() > xr * half_tan
        nb = torch.where(out, (cand + torch.where(y > 0, 1, -1)) % 18, cand)
        u2, y2, l2 = cross(nb, xr)
        u, y, l, cand = torch.where(out, u2, u), torch.where(out, y2, y), torch.where(out, l2, l), nb
        z = z0 + tanl * l
        alive &= (u.abs() < 0.99) & (y.abs() <= xr * half_tan) & (l > l_prev) & (z.abs() <= 250.0)
        l_prev = torch.where(alive, l, l_prev)
        hy[r], hz[r], hs[r], keep[r] = y, z, cand + torch.where(z < 0, 18, 0), alive & ~drop[r]
    if lengths == "capped":
        cap = torch.randint(10, ROWS + 1, (n,), generator=gen, device=DEV)
        keep &= torch.cumsum(keep, 0) <= cap
    keep &= keep.sum(0) >= 10
    if d_true is not None:
        d = d_true.to(F64)[hs, torch.arange(ROWS, device=DEV)[:, None]]
        hy, hz = hy + d[..., 0], hz + d[..., 1]
    return hy, hz, hs, keep


def _tracks(n, seed, lengths, d_true=None):
    """n fitted-for tracks as device tensors: y, z, rowsec, offsets, seeds."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    parts, got = [], 0
    while got < n:
        m = min(200_000, int((n - got) * 1.03) + 64)
        hy, hz, hs, keep = _simulate(m, gen, lengths, d_true)
        good = keep.any(0).nonzero()[: n - got, 0]
        kt = keep[:, good].t().contiguous()
        trk, row = kt.nonzero(as_tuple=True)
        col = good[trk]
        y = hy[row, col] + 0.1 * torch.randn(row.numel(), generator=gen, device=DEV, dtype=F64)
        z = hz[row, col] + 0.1 * torch.randn(row.numel(), generator=gen, device=DEV, dtype=F64)
        parts.append((y.float(), z.float(), (row << 6 | hs[row, col]), kt.sum(1)))
        got += good.numel()
    y, z, rs, count = (torch.cat([p[i] for p in parts]) for i in range(4))
    y, z, rs, count = _thin(n, gen, lengths, y, z, rs, count)
    off = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    torch.cumsum(count, 0, out=off[1:])
    rowsec = torch.where(rs >= 1 << 15, rs - (1 << 16), rs).to(torch.int16)
    return dict(y=y, z=z, rowsec=rowsec, offsets=off.to(torch.int32), seeds=_seeds(y, z, rs, off).float().contiguous())


def _hits(n, lengths):
    """Clusters of n tracks: a little below the expected number, by four times what it varies by."""
    return int(n * MEAN_HITS[lengths] * (1.0 - {"natural": 0.06, "capped": 2.1}[lengths] / math.sqrt(n + 16)))


def _thin(n, gen, lengths, y, z, rs, count):
    """As many clusters for every seed: a random few more are lost, none of a track's first ten."""
    extra = y.numel() - _hits(n, lengths)
    if extra <= 0:
        raise ValueError("fewer clusters than expected")
    owner = torch.repeat_interleave(torch.arange(n, device=DEV), count)
    place = torch.arange(y.numel(), device=DEV) - (torch.cumsum(count, 0) - count)[owner]
    rank = torch.rand(y.numel(), generator=gen, device=DEV, dtype=F64) + (place < 10)
    lost = torch.topk(rank, extra, largest=False).indices
    keep = torch.ones(y.numel(), device=DEV, dtype=torch.bool)
    keep[lost] = False
    return y[keep], z[keep], rs[keep], torch.bincount(owner[keep], minlength=n)


def _seeds(y, z, rs, off):
    """Circle through the first, middle and last cluster (the recipe of synth.three_point_seeds)."""
    first, last = off[:-1], off[1:] - 1
    row_x = torch.as_tensor(synth.default_geometry().row_x, device=DEV)

    def point(i):
        a = ((rs[i] & 63) % 18 + 0.5) * math.radians(20.0)
        x = row_x[rs[i] >> 6]
        yy = y[i].to(F64)
        return x * torch.cos(a) - yy * torch.sin(a), x * torch.sin(a) + yy * torch.cos(a), a

    x0, y0, a0 = point(first)
    x1, y1, _ = point(first + (last - first) // 2)
    x2, y2, _ = point(last)
    l01, l12, l02 = torch.hypot(x1 - x0, y1 - y0), torch.hypot(x2 - x1, y2 - y1), torch.hypot(x2 - x0, y2 - y0)
    turn = (x1 - x0) * (y2 - y1) - (y1 - y0) * (x2 - x1)
    kappa = synth.KAPPA_PER_TESLA * 0.5
    k = 2.0 * turn / (l01 * l12 * l02)
    k = torch.where(k.abs() < 1e-12, 1e-4 * abs(kappa), k)
    phi = torch.atan2(y1 - y0, x1 - x0) - torch.asin((k * l01 * 0.5).clamp(-1, 1))
    arc = 2.0 * torch.asin((k.abs() * l02 * 0.5).clamp(0, 1)) / k.abs()
    z0, z2 = z[first].to(F64), z[last].to(F64)
    return torch.stack([y[first].to(F64), z0, torch.sin(phi - a0), (z2 - z0) / arc, k / kappa])


def _offsets(seed, n=1, sigma=0.05):
    """n tables of alignment offsets N(0, 0.05 cm), [n, 36, 152, 2]."""
    gen = torch.Generator(device=DEV).manual_seed(seed + 7)
    return sigma * torch.randn((n, 36, ROWS, 2), generator=gen, device=DEV)


def _frame_sizes(case):
    """Tracks per frame: log-uniform, of one expected total, the same for every seed."""
    rng = np.random.default_rng(1000 * case["frames"] + case["lo"])
    sizes = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]), case["frames"])).astype(np.int64)
    total = case["frames"] * (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
    return np.maximum(1, (sizes * (total / sizes.sum())).astype(np.int64))


def _inputs(case, seed):
    """Everything a pass reads, without the library."""
    if case["kind"] == "frames":
        sizes = _frame_sizes(case)
        base = torch.from_numpy(np.concatenate([[0], np.cumsum(sizes)])).to(DEV)
        d = _tracks(int(sizes.sum()), seed, "capped")
        return dict(d, frame_base=base, frame_alignment=_offsets(seed, case["frames"]))
    table = _offsets(seed)[0] if case.get("align") else None
    d = _tracks(case["tracks"], seed, case["lengths"], table)
    d["align"] = table
    if case["kind"] in ("adjoint", "adjoint_host"):
        # weights of the tracks in the objective sum_i g_i chi2_i
        gen = torch.Generator(device=DEV).manual_seed(seed + 3)
        d["grad_chi2"] = 0.5 + torch.rand(case["tracks"], generator=gen, device=DEV)
    if case["kind"] == "reject":
        # leave-one-out chi2 of good clusters (2 degrees of freedom), and 2% of them beyond the cut
        gen = torch.Generator(device=DEV).manual_seed(seed + 5)
        h = d["y"].numel()
        u = 1e-3 + 0.999 * torch.rand(h, generator=gen, device=DEV)
        far = torch.zeros(h, device=DEV, dtype=torch.bool)
        far[torch.randperm(h, generator=gen, device=DEV)[: h // 50]] = True
        d["chi2"] = torch.where(far, 16.5 - 40.0 * torch.log(u), -2.0 * torch.log(u))
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    f = tf.Fitter(synth.default_geometry(), 0.5, deterministic=bool(case.get("det")))
    f.set_material(GAS if case.get("material") else None)
    f.set_field(FIELD if case.get("field") else None)
    if d.get("align") is not None:
        f.set_alignment(d["align"].reshape(-1))
    f.set_record(case["kind"] in ("adjoint", "smooth", "states"))
    s = dict(case=case, f=f, d=d)
    n = int(d["offsets"].numel()) - 1
    if case["kind"] == "frames":
        s["batch"] = FrameBatch(d["y"], d["z"], d["rowsec"], d["offsets"], d["seeds"], d["frame_base"])
    if case["kind"] == "adjoint_host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        s["host"] = [pin(d["y"]), pin(d["z"]), pin(d["rowsec"]).numpy().view(np.uint16), pin(d["offsets"]),
                     pin(d["seeds"]), pin(d["grad_chi2"])]
        s["back"] = dict(chi2=torch.empty(n).pin_memory(), ndf=torch.empty(n, dtype=torch.int32).pin_memory(),
                         grad_align=torch.empty((36, ROWS, 2)).pin_memory(), grad_seeds=torch.empty((5, n)).pin_memory())
        d.clear()
    else:
        s["out"] = tf.empty_outputs(n)
        if case.get("meas"):
            s["meas"] = torch.empty((d["y"].numel(), 2), device=DEV)
    torch.cuda.synchronize()
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    f, d, kind = s["f"], s["d"], s["case"]["kind"]
    if kind == "fit":
        return f.fit(d, s["out"])
    if kind == "frames":
        return fit_frames(f, s["batch"], s["out"], d["frame_alignment"])
    if kind == "adjoint":
        out = f.fit(d, s["out"])
        ga, gs = f.backward(d, out, d["grad_chi2"], s.get("meas"))
        r = dict(out, grad_align=ga, grad_seeds=gs)
        return dict(r, grad_meas=s["meas"]) if "meas" in s else r
    if kind == "adjoint_host":
        return tf.tpcfit_fit_adjoint_host(f.h, *s["host"], out=s["back"])
    if kind == "smooth":
        out = f.fit(d, s["out"])
        return f.smooth(d, out)
    if kind == "states":
        out = f.fit(d, s["out"])
        return f.smooth_states(d, out)
    r = f.reject_outliers(d, d["chi2"], 16.0)
    return {k: r[k] for k in ("y", "z", "rowsec", "offsets")}


def _sizes(case):
    if case["kind"] == "frames":
        n = int(_frame_sizes(case).sum())
        return n, _hits(n, "capped")
    return case["tracks"], _hits(case["tracks"], case["lengths"])


def work(case):
    """Each input read once, each output written once; the operations of the filter in U-D form per cluster and
    pass (257), of its reverse (656), of the combination of the two filters (about 400 for the residual, 700 for the
    state).  The reproducible mode and the material layers need the square-root form: 397, 806 and about 330 for a
    layer."""
    n, h = _sizes(case)
    kind = case["kind"]
    sqrt_form = case.get("det") or case.get("material")
    step = 397 if sqrt_form else 257
    step += 330 if case.get("material") else 0
    fit_bytes, fit_out, fit_flops = 10 * h + 24 * n, 88 * n, 2 * step * h
    if kind in ("fit", "frames"):
        return dict(bytes=fit_bytes + fit_out, flops=fit_flops)
    if kind in ("adjoint", "adjoint_host"):
        rev = 2 * (806 if sqrt_form else 656) * h
        grads = 4 * n + 20 * n + 43_776 + (8 * h if case.get("meas") else 0)
        return dict(bytes=fit_bytes + (fit_out if kind == "adjoint" else 8 * n) + grads, flops=fit_flops + rev)
    if kind == "smooth":
        return dict(bytes=fit_bytes + 24 * h, flops=fit_flops + 400 * h)
    if kind == "states":
        return dict(bytes=fit_bytes + 80 * h, flops=fit_flops + 700 * h)
    return dict(bytes=24 * h + 8 * n, flops=0)


# ---------------------------------------------------------------- the filter at 64 bits
class _Filter:
    """The extended Kalman filter of some tracks at 64 bits, covariance form: states p [n, 5] = (y, z, sin phi,
    tan lambda, q/pt) and covariances C [n, 5, 5]; clusters step by step over a padded [n, steps] layout."""

    MAX_SNP = float(np.float32(0.999))
    V = float(np.float32(0.01))

    def __init__(self, case, y, z, rowsec, off, seeds, table):
        rs = rowsec.to(torch.int64) & 0xFFFF
        n = off.numel() - 1
        self.n, self.len = n, off[1:] - off[:-1]
        self.steps = int(self.len.max())
        j = torch.arange(self.steps, device=DEV)
        self.has = j[None, :] < self.len[:, None]
        self.hit = torch.where(self.has, off[:-1, None] + j[None, :], off[:-1, None])
        row, sec = rs >> 6, rs & 63
        m = torch.stack([y, z], 1).to(F64)
        if table is not None:
            m = m - (table(sec, row)).to(F64)
        self.m = [t.clone() for t in m[self.hit].unbind(1)]  # measured (y, z), alignment taken off
        x = torch.as_tensor(synth.default_geometry().row_x, device=DEV).float().to(F64)
        self.x = x[row[self.hit]].unbind(1)
        self.sec = (sec % 18)[self.hit].unbind(1)
        self.seed = seeds.to(F64).t().contiguous()
        self.kappa = float(np.float32(synth.KAPPA_PER_TESLA * 0.5))
        self.mat = GAS if case.get("material") else None
        self.fld = FIELD if case.get("field") else None
        a = np.arange(18)
        t = np.deg2rad(20.0 * (((a[None, :] - a[:, None]) % 18 + 8) % 18 - 8))
        self.cos = torch.as_tensor(np.cos(t).astype(np.float32), device=DEV).to(F64)
        self.sin = torch.as_tensor(np.sin(t).astype(np.float32), device=DEV).to(F64)
        self.c0 = 100.0 * torch.eye(5, device=DEV, dtype=F64).expand(n, 5, 5)

    def layer(self, p, direction):
        """A row's material layer: the state after it, the scale of q and the noise."""
        g = self.mat
        s, t, q = p[:, 2], p[:, 3], p[:, 4]
        tt = 1.0 + t * t
        c, st = torch.sqrt((1.0 - s) * (1.0 + s)), torch.sqrt(tt)
        ell = g.row_cm * st / c
        p2 = tt / (q * q)
        e2 = p2 + g.mass_gev ** 2
        th = torch.sqrt(0.0136 ** 2 * ell / g.x0_cm * e2 / (p2 * p2))
        de = g.dedx_gev_cm * ell * e2 / p2
        pn2 = (torch.sqrt(e2) - direction * de) ** 2 - g.mass_gev ** 2
        qq = torch.sqrt(p2 / pn2)
        qn = q * qq
        zero = torch.zeros_like(q)
        b1 = torch.stack([zero, zero, th * c * st, zero, zero], 1)
        b2 = torch.stack([zero, zero, zero, th * tt, th * qn * t], 1)
        noise = b1[:, :, None] * b1[:, None, :] + b2[:, :, None] * b2[:, None, :]
        return torch.cat([p[:, :4], qn[:, None]], 1), qq, noise

    @staticmethod
    def scatter(C, qq, noise):
        one = torch.ones_like(qq)
        d = torch.stack([one, one, one, one, qq], 1)
        return C * d[:, :, None] * d[:, None, :] + noise

    def move(self, p, x, a, b, X):
        """Propagation to X in the frame of sector b: the state, its Jacobian, and where it is possible."""
        rot = a != b
        ca, sa = self.cos[a, b], self.sin[a, b]
        y, z, s, t, q = p.unbind(1)
        c = torch.sqrt((1.0 - s) * (1.0 + s))
        sr, cr = s * ca - c * sa, c * ca + s * sa
        x1 = torch.where(rot, x * ca + y * sa, x)
        y1 = torch.where(rot, y * ca - x * sa, y)
        s1 = torch.where(rot, sr, s)
        ok = (cr > 0) & (s1.abs() < self.MAX_SNP)
        s1 = torch.where(ok, s1, torch.zeros_like(s1))
        dx = X - x1
        kappa = self.kappa
        if self.fld is not None:
            c1 = torch.sqrt((1.0 - s1) * (1.0 + s1))
            xm, ym, zm = x1 + 0.5 * dx, y1 + 0.5 * dx * s1 / c1, z + 0.5 * dx * t / c1
            kappa = kappa * (1.0 + self.fld.c_r / 250.0 ** 2 * (xm * xm + ym * ym) + self.fld.c_z / 250.0 ** 2 * zm * zm)
        k = q * kappa
        kdx = k * dx
        s2 = s1 + kdx
        ok = ok & (s2.abs() < self.MAX_SNP)
        s2 = torch.where(ok, s2, s1)
        ic1, ic2 = 1.0 / torch.sqrt((1.0 - s1) * (1.0 + s1)), 1.0 / torch.sqrt((1.0 - s2) * (1.0 + s2))
        tm = (s1 + s2) / (1.0 / ic1 + 1.0 / ic2)
        w = 1.0 / ic1 + s1 * tm
        sig = torch.where(ok, kdx * w, torch.zeros_like(w))
        tiny = sig.abs() < 1e-4
        sg = torch.where(tiny, torch.ones_like(sig), sig)
        dl = dx * w * torch.where(tiny, 1.0 + sig * sig / 6.0 + 0.075 * sig ** 4, torch.asin(sg.clamp(-1, 1)) / sg)
        small = kdx.abs() < 1e-3
        ks = torch.where(small, torch.ones_like(k), k)
        i3 = ic1 ** 3
        series = dx * dx * (0.5 * s1 * i3 + kdx * ((1 + 2 * s1 * s1) * ic1 ** 5 / 3 + kdx * (
            s1 * (3 + 2 * s1 * s1) * ic1 ** 7 / 8 + kdx * (3 + 24 * s1 * s1 + 8 * s1 ** 4) * ic1 ** 9 / 30)))
        lk = torch.where(small, series, (dx * ic2 - dl) / ks)
        tt = 1.0 + tm * tm
        ys, yq = dx * tt * (ic1 + ic2) * 0.5, dx * kappa * dx * tt * ic2 * 0.5
        zs, zt, zq, sq = t * dx * tm * ic1 * ic2, dl, t * kappa * lk, dx * kappa
        one, zero = torch.ones_like(s), torch.zeros_like(s)
        rr = torch.where(rot, cr / c, one)
        yy = torch.where(rot, ca - sa * s2 * ic2, one)
        zy = torch.where(rot, -sa * t * ic2, zero)
        sy = torch.where(rot, -sa * k, zero)
        J = torch.stack([yy, zero, ys * rr, zero, yq, zy, one, zs * rr, zt, zq, sy, zero, rr, zero, sq,
                         zero, zero, zero, one, zero, zero, zero, zero, zero, one], 1).view(-1, 5, 5)
        return torch.stack([y1 + dx * tm, z + t * dl, s2, t, q], 1), J, ok

    def update(self, p, C, m):
        chi2 = 0.0
        for h in (0, 1):
            S = C[:, h, h] + self.V
            K = C[:, :, h] / S[:, None]
            r = m[:, h] - p[:, h]
            p = p + K * r[:, None]
            C = C - K[:, :, None] * C[:, h, None, :]
            chi2 = chi2 + r * r / S
        return p, C, chi2

    def passes(self, predicted=None, filtered=None):
        """Outward pass and inward refit; predicted(direction, j, p, C, at) and filtered(...) see the states."""
        n = self.n
        p = self.seed
        last = torch.full((n,), -1, device=DEV)
        alive = torch.ones(n, device=DEV, dtype=torch.bool)
        failed = torch.zeros(n, device=DEV, dtype=torch.bool)
        chi2 = torch.zeros(n, device=DEV, dtype=F64)
        for direction in (1, -1):
            C = self.c0
            xs = torch.zeros(n, device=DEV, dtype=F64)
            secs = torch.zeros(n, device=DEV, dtype=torch.int64)
            chi2 = torch.zeros(n, device=DEV, dtype=F64)
            for j in (range(self.steps) if direction > 0 else range(self.steps - 1, -1, -1)):
                if direction > 0:
                    at, first = alive & self.has[:, j], torch.full_like(alive, j == 0)
                else:
                    at, first = (last >= j) & ~failed, last == j
                pb, Cb = p, C
                step = at & ~first
                go = at
                if not bool(first.all()):
                    if self.mat is not None and direction < 0:
                        pb, qq, noise = self.layer(pb, -1)
                        Cb = self.scatter(Cb, qq, noise)
                    # tracks that take no step here go through with a harmless one
                    px = torch.where(step[:, None], pb, self.safe)
                    xf = torch.where(step, xs, self.x[j] - 1.0)
                    sf = torch.where(step, secs, self.sec[j])
                    pn, J, ok = self.move(px, xf, sf, self.sec[j], self.x[j])
                    Cn = J @ Cb @ J.transpose(1, 2)
                    if self.mat is not None and direction > 0:
                        pn, qq, noise = self.layer(pn, 1)
                        Cn = self.scatter(Cn, qq, noise)
                    go = at & (first | ok)
                    if direction > 0:
                        alive = alive & ~(step & ~ok)
                    else:
                        failed = failed | (step & ~ok)
                    moved = (step & ok)
                    pb = torch.where(moved[:, None], pn, p)
                    Cb = torch.where(moved[:, None, None], Cn, C)
                if predicted is not None:
                    predicted(direction, j, pb, Cb, go)
                pu, Cu, dc = self.update(pb, Cb, self.m[j])
                p = torch.where(go[:, None], pu, p)
                C = torch.where(go[:, None, None], Cu, C)
                chi2 = chi2 + torch.where(go, dc, torch.zeros_like(dc))
                xs, secs = torch.where(go, self.x[j], xs), torch.where(go, self.sec[j], secs)
                if direction > 0:
                    last = torch.where(go, j, last)
                if filtered is not None:
                    filtered(direction, j, p, C, go)
        self.last = last
        good = ~failed & (last >= 2)
        ndf = torch.where(good, 2 * (last + 1) - 5, -1)
        return p, C, chi2, ndf, good

    safe = None

    def fit(self):
        p, C, chi2, ndf, good = self.passes()
        nan = torch.full((), math.nan, device=DEV, dtype=F64)
        i, j = torch.tril_indices(5, 5, device=DEV)
        return dict(params=torch.where(good, p.t(), nan), cov=torch.where(good, C[:, i, j].t(), nan),
                    chi2=torch.where(good, chi2, nan), ndf=ndf)


def _filter(case, d, lo, hi):
    off = d["offsets"].to(torch.int64)
    h0, h1 = int(off[lo]), int(off[hi])
    table = None
    if case["kind"] == "frames":
        fa = d["frame_alignment"]
        frame = torch.searchsorted(d["frame_base"], torch.arange(lo, hi, device=DEV), right=True) - 1
        owner = torch.repeat_interleave(frame, off[lo + 1:hi + 1] - off[lo:hi])
        table = lambda sec, row: fa[owner, sec, row]  # noqa: E731
    elif d.get("align") is not None:
        table = lambda sec, row: d["align"][sec, row]  # noqa: E731
    F = _Filter(case, d["y"][h0:h1], d["z"][h0:h1], d["rowsec"][h0:h1], off[lo:hi + 1] - h0, d["seeds"][:, lo:hi], table)
    F.safe = torch.tensor([0.0, 0.0, 0.0, 0.0, 1.0], device=DEV, dtype=F64).expand(hi - lo, 5)
    return F, h0, h1


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    n, H = int(d["offsets"].numel()) - 1, int(d["y"].numel())
    if kind == "reject":
        keep = ~(d["chi2"] > 16.0)
        count = torch.cat([torch.zeros(1, device=DEV, dtype=torch.int64), torch.cumsum(keep, 0)])
        return dict(y=d["y"][keep].to(F64), z=d["z"][keep].to(F64), rowsec=d["rowsec"][keep],
                    offsets=count[d["offsets"].to(torch.int64)].to(torch.int32))
    out = {k: [] for k in ("params", "cov", "chi2", "ndf", "grad_seeds")}
    gm = torch.zeros((H, 2), device=DEV, dtype=F64)
    sm = {}
    chunk = {"smooth": 100_000, "states": 50_000, "adjoint": 50_000, "adjoint_host": 50_000}.get(kind, 200_000)
    for lo in range(0, n, chunk):
        F, h0, h1 = _filter(case, d, lo, min(n, lo + chunk))
        if kind in ("adjoint", "adjoint_host"):
            _gradients(F, d["grad_chi2"][lo:lo + chunk].to(F64), out, gm[h0:h1])
        elif kind in ("smooth", "states"):
            for k, v in _smoothed(F, kind, h1 - h0).items():
                sm.setdefault(k, []).append(v)
        else:
            for k, v in F.fit().items():
                out[k].append(v)
    if sm:
        return {k: torch.cat(v) for k, v in sm.items()}
    r = {k: torch.cat(v, -1) for k, v in out.items() if v}
    r["ndf"] = r["ndf"].to(torch.int32)
    if kind in ("adjoint", "adjoint_host"):
        rs = d["rowsec"].to(torch.int64) & 0xFFFF
        ga = torch.zeros((36 * ROWS, 2), device=DEV, dtype=F64)
        ga.index_add_(0, (rs & 63) * ROWS + (rs >> 6), gm)
        r["grad_align"] = -ga.view(36, ROWS, 2)
        if case.get("meas"):
            r["grad_meas"] = gm
    return r if kind != "adjoint_host" else {k: r[k] for k in ("chi2", "ndf", "grad_align", "grad_seeds")}


def _gradients(F, g, out, gm):
    F.seed = F.seed.requires_grad_()
    F.m = [t.requires_grad_() for t in F.m]
    with torch.enable_grad():
        r = F.fit()
        loss = (g * torch.where(r["ndf"] > 0, r["chi2"], torch.zeros_like(g))).sum()
    grads = torch.autograd.grad(loss, [F.seed, *F.m])
    for k, v in r.items():
        out[k].append(v.detach())
    out["grad_seeds"].append(grads[0].t())
    per = torch.stack(grads[1:], 1)
    gm[F.hit[F.has]] = per[F.has]


def _smoothed(F, kind, hits):
    """Two-filter smoother: the outward estimate (without the cluster's own update for the residuals, with it for the
    states) combined with the inward prediction."""
    outward = {}
    nan = math.nan
    if kind == "smooth":
        r = dict(resid=torch.full((hits, 2), nan, device=DEV, dtype=F64), rcov=torch.full((hits, 3), nan, device=DEV, dtype=F64),
                 chi2=torch.full((hits,), nan, device=DEV, dtype=F64))
    else:
        r = dict(state=torch.full((hits, 5), nan, device=DEV, dtype=F64), state_cov=torch.full((hits, 15), nan, device=DEV, dtype=F64))
    tri = torch.tril_indices(5, 5, device=DEV)

    def outgoing(direction, j, p, C, at):
        if direction > 0:
            outward[j] = (p, C)

    def predicted(direction, j, p, C, at):
        if direction > 0:
            if kind == "smooth":
                outward[j] = (p, C)
            return
        po, Co = outward.pop(j)
        # of p.d. sum S: gain = Co S^-1
        gain = torch.linalg.solve(Co + C, Co).transpose(1, 2)
        x = po + (gain @ (p - po)[:, :, None])[:, :, 0]
        Cs = gain @ C
        Cs = 0.5 * (Cs + Cs.transpose(1, 2))
        h = F.hit[at, j]
        if kind == "states":
            r["state"][h] = x[at]
            r["state_cov"][h] = Cs[:, tri[0], tri[1]][at]
            return
        res = F.m[j] - x[:, :2]
        R = Cs[:, :2, :2] + F.V * torch.eye(2, device=DEV, dtype=F64)
        c2 = (res[:, None, :] @ torch.linalg.solve(R, res[:, :, None]))[:, 0, 0]
        r["resid"][h] = res[at]
        r["rcov"][h] = torch.stack([R[:, 0, 0], R[:, 1, 0], R[:, 1, 1]], 1)[at]
        r["chi2"][h] = c2[at]

    _, _, _, _, good = F.passes(predicted, outgoing if kind == "states" else None)
    bad = (~good[:, None] & F.has)
    for v in r.values():
        v[F.hit[bad]] = nan
    return r
