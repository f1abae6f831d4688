"""The calls whose time matters to a user of libptycho, as cases to be timed.

``listed()`` names them, ``draw(rng)`` makes more of the same ranges,
``prepare`` builds what a reconstruction program holds before the call (data,
current object and probe, the handle), ``run`` is the call itself through the
package's public entry points, ``work`` the bytes and operations it cannot do
without, and ``exact`` the same results in 64 bits from plain torch.

The inputs are those of a reconstruction under way: a scan over a textured
object, Poisson counts of its far field (or of its propagated wave), and an
object and probe estimate near but not at the solution, so that the model's
far field is filled as it is after the first cycles.
"""
import math

import numpy as np
import torch

from paper_2008_11511_gb300 import Ptycho, PtychoBatch, fft2

# frame sizes by use: powers of two, detector crops with factors 3, 5 and 7
SIZES_ONE_MODE = (64, 80, 128, 160, 192, 224, 256, 384, 400, 448, 512)
SIZES_MODES = (128, 192, 256, 384, 512)


def listed():
    return [
        # the smallest reconstruction: a quick-look scan of 100 small frames, a few
        # alternating-projection cycles per call (launch and latency bound)
        dict(name="ap64", kind="ap", N=64, K=1, J=100, Ho=256, Wo=256, cycles=5, mask=False, photons=1e5),
        # the standard large scan: difference-map cycles on 4000 frames of 256^2 with
        # a detector-gap mask, one cycle per call (the headline workload)
        dict(name="dm256", kind="dm", N=256, K=1, J=4000, Ho=2048, Wo=2048, cycles=1, mask=True, photons=1e6),
        # partially coherent illumination: three probe modes on 512^2 frames
        dict(name="dm512_modes", kind="dm", N=512, K=3, J=300, Ho=1700, Wo=1700, cycles=1, mask=True, photons=1e7),
        # detector crop of 400^2, ragged frame count and object, incoherent
        # background refined along with object and probe
        dict(name="ap400_bg", kind="ap", N=400, K=1, J=203, Ho=1333, Wo=1201, cycles=1, mask=True, photons=1e6,
             background=True),
        # near-field scan: projection on the propagated wave
        dict(name="nf256", kind="dm", N=256, K=1, J=500, Ho=1100, Wo=1100, cycles=1, mask=True, photons=1e8,
             nearfield=200.0),
        # one gradient of the Poisson likelihood for an outside optimiser, object and probe
        dict(name="grad256", kind="grad", N=256, K=1, J=1000, Ho=1536, Wo=1536, mask=True, photons=1e5),
        # refinement after the projection cycles: conjugate-gradient steps on the object
        dict(name="cg256", kind="cg", N=256, K=1, J=1000, Ho=1536, Wo=1536, cycles=2, mask=True, photons=1e6,
             update_probe=False),
        # the same refinement of object and probe with three modes
        dict(name="cg256_modes", kind="cg", N=256, K=3, J=150, Ho=900, Wo=901, cycles=1, mask=True, photons=1e6,
             update_probe=True),
        # the likelihood alone, as monitored between steps, on many small frames
        dict(name="llk128", kind="llk", N=128, K=1, J=2500, Ho=1024, Wo=1024, mask=True, photons=1e5),
        # several scans of different frame sizes reconstructed side by side in one handle
        dict(name="batch", kind="batch", sizes="128:301,192:97,256:210,384:61,512:50,64:150", mask=True,
             photons=1e5, cycles=1),
        # the transform operator by itself, in place on a stack of frames
        dict(name="fft256", kind="fft", N=256, J=1024, direction=-1),
        # position refinement: the per-frame shifts after a projection cycle
        dict(name="pos256", kind="pos", N=256, K=1, J=1000, Ho=1536, Wo=1536, mask=False, photons=1e6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("ap", "dm", "dm", "dm_modes", "nf", "grad", "cg", "cg_modes", "llk", "batch", "fft", "pos"))
    photons = 10.0 ** rng.uniform(5, 7)
    if kind == "batch":
        n = rng.randint(2, 8)
        parts = []
        for _ in range(n):
            N = rng.choice((64, 128, 192, 256, 384, 512))
            parts.append("%d:%d" % (N, _log_int(rng, 20, max(21, 1.2e7 / (N * N)))))
        return dict(kind="batch", sizes=",".join(parts), mask=rng.random() < 0.5, photons=10.0 ** rng.uniform(4.5, 6),
                    cycles=1)
    if kind == "fft":
        N = rng.choice((16, 32) + SIZES_ONE_MODE)
        return dict(kind="fft", N=N, J=_log_int(rng, 8, min(20000, 6.4e7 / (N * N))), direction=rng.choice((-1, 1)))
    modes = kind.endswith("_modes")
    K = rng.choice((2, 3)) if modes else 1
    N = rng.choice(SIZES_MODES if modes else SIZES_ONE_MODE)
    # frames x modes x pixels: from a small scan to about half of the largest listed one
    most = {"dm": 1.2e8, "ap": 1.2e8, "dm_modes": 1.2e8, "nf": 6e7, "llk": 1.2e8}.get(kind, 4e7)
    J = _log_int(rng, 25, max(26, min(6000, most / (K * N * N))))
    # neighbouring frames a tenth to a fifth of a frame apart; the object just covers the scan
    side = N + int(rng.uniform(0.08, 0.2) * N * math.sqrt(J)) + 2
    case = dict(kind=kind.split("_")[0], N=N, K=K, J=J, Ho=side + rng.randint(0, 9), Wo=side + rng.randint(0, 9),
                mask=rng.random() < 0.6, photons=photons)
    if kind == "nf":
        case.update(kind="dm", nearfield=rng.uniform(0.3, 1.0) * N, photons=photons * 100)
    if case["kind"] in ("ap", "dm"):
        case["cycles"] = rng.randint(1, 3)
        if case["kind"] == "ap" and rng.random() < 0.4:
            case["background"] = True
    if case["kind"] == "cg":
        case.update(cycles=rng.randint(1, 2), update_probe=rng.random() < 0.5)
    if case["kind"] in ("grad", "cg"):
        case["photons"] = min(photons, 1e6)
    return case


# ---------------------------------------------------------------- inputs


def _problems(case):
    """The scans of a case: one, or those of a batch."""
    if case["kind"] != "batch":
        return [case]
    out = []
    for i, part in enumerate(case["sizes"].split(",")):
        N, J = (int(v) for v in part.split(":"))
        side = N + int(0.12 * N * math.sqrt(J)) + 3
        out.append(dict(kind="dm" if i % 2 else "ap", N=N, K=1, J=J, Ho=side, Wo=side + i % 3, cycles=case["cycles"],
                        mask=case["mask"], photons=case["photons"]))
    return out


def _positions(J, N, Ho, Wo, seed):
    """Fermat spiral over the object with a pixel of jitter."""
    r = np.random.default_rng(seed)
    m = np.arange(J)
    rad, ang = np.sqrt((m + 0.5) / J), np.deg2rad(137.508) * m
    y = (Ho - N) / 2 * (1 + rad * np.sin(ang)) + r.uniform(-1, 1, J)
    x = (Wo - N) / 2 * (1 + rad * np.cos(ang)) + r.uniform(-1, 1, J)
    pos = np.stack([np.clip(np.rint(y), 0, Ho - N), np.clip(np.rint(x), 0, Wo - N)], axis=1)
    return np.ascontiguousarray(pos.astype(np.int32))


def _mask(N):
    """Two dead bands of a tiled detector, about 2 % of the pixels, in FFT order."""
    m = np.zeros((N, N), dtype=np.uint8)
    w = max(1, N // 64)
    m[N // 2 + N // 8:N // 2 + N // 8 + w, :] = 1
    m[:N // 3, N // 2 - N // 5:N // 2 - N // 5 + w] = 1
    return np.fft.ifftshift(m)


def _noise(shape, g):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda"))


def _smooth(shape, sigma, g):
    """Real Gaussian random field of unit spread, correlated over `sigma` pixels."""
    ky = torch.fft.fftfreq(shape[0], device="cuda")[:, None]
    kx = torch.fft.fftfreq(shape[1], device="cuda")[None, :]
    f = torch.fft.fft2(torch.randn(*shape, generator=g, device="cuda")) * torch.exp(-2 * (math.pi * sigma) ** 2 * (ky ** 2 + kx ** 2))
    f = torch.fft.ifft2(f).real
    return f / f.std()


def _probe(case, g):
    """Aperture with a quadratic phase (far field), a wide diffuse beam (near
    field), or Hermite-Gauss modes of falling weight."""
    N, K = case["N"], case["K"]
    t = torch.arange(N, device="cuda", dtype=torch.float32) - N / 2
    y, x = t[:, None], t[None, :]
    r2 = y * y + x * x
    if K == 1:
        near = bool(case.get("nearfield"))
        rad = N * (0.35 if near else 0.17)
        amp = torch.sigmoid((rad - r2.sqrt()) * 1.5)
        ph = 0.24 / rad * r2 + (2.0 * _smooth((N, N), 4.0, g) if near else 0.0)
        return (amp * torch.exp(1j * ph))[None]
    s = N * 0.12
    env = torch.exp(-r2 / (2 * s * s)) * torch.exp(1j * (0.24 / s) * r2 / 2)
    herm = [torch.ones_like(r2), x / s, y / s, x * y / (s * s)]
    out = []
    for k in range(K):
        m = env * herm[k % 4]
        out.append(m / m.abs().square().sum().sqrt() * math.sqrt((0.7, 0.2, 0.1, 0.05)[k % 4]))
    return torch.stack(out)


def _patches(obj, pos, N, lo, hi):
    """obj[r_j + y, c_j + x] for frames lo .. hi - 1."""
    t = torch.arange(N, device=obj.device)
    p = torch.as_tensor(pos[lo:hi].astype(np.int64), device=obj.device)
    return obj[(p[:, 0, None] + t)[:, :, None], (p[:, 1, None] + t)[:, None, :]]


def _chunks(case, most=1 << 25):
    n = max(1, most // (case["K"] * case["N"] ** 2))
    for lo in range(0, case["J"], n):
        yield lo, min(case["J"], lo + n)


def _transfer(case, dtype):
    """Near-field propagator exp(-i pi c (ky^2 + kx^2) / N^2), or None in the far field."""
    c, N = case.get("nearfield"), case["N"]
    if not c:
        return None
    k = torch.fft.fftfreq(N, device="cuda", dtype=torch.float64) * N
    return torch.exp(-1j * math.pi * c * (k[:, None] ** 2 + k[None, :] ** 2) / N ** 2).to(dtype)


def _detect(wave, h):
    f = torch.fft.fft2(wave, norm="ortho")
    return f if h is None else torch.fft.ifft2(f * h, norm="ortho")


def _undetect(wave, h):
    return torch.fft.ifft2(wave, norm="ortho") if h is None else torch.fft.ifft2(torch.fft.fft2(wave, norm="ortho") * h.conj(), norm="ortho")


def _scan(case, seed):
    """Data, positions, mask and the current estimates of one scan."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    N, K, J, Ho, Wo = (case[k] for k in ("N", "K", "J", "Ho", "Wo"))
    pos = _positions(J, N, Ho, Wo, seed)
    mask = _mask(N) if case["mask"] else None
    true = (0.9 + 0.05 * _smooth((Ho, Wo), 3.0, g)) * torch.exp(0.8j * _smooth((Ho, Wo), 4.0, g)) + 0.04 * _noise((Ho, Wo), g)
    probe = _probe(case, g)
    probe = probe * math.sqrt(case["photons"] / float(probe.abs().square().sum()) / 0.81)
    h = _transfer(case, torch.complex64)
    bg = None
    if case.get("background"):
        bg = case["photons"] / (N * N) * 0.02 * (1 + 0.2 * _smooth((N, N), N / 16, g)).clamp_min(0.1)
    iobs = torch.empty((J, N, N), device="cuda")
    for lo, hi in _chunks(case):
        lam = _detect(_patches(true, pos, N, lo, hi)[:, None] * probe, h).abs().square().sum(1)
        iobs[lo:hi] = torch.poisson(lam if bg is None else lam + bg, generator=g)
    if mask is not None:
        iobs[:, torch.as_tensor(mask, device="cuda") != 0] = 0
    # gradient steps refine what the projection cycles have brought near the solution
    e = 0.005 if case["kind"] in ("grad", "cg") else 1.0
    obj = (true * torch.exp(0.15j * e * _smooth((Ho, Wo), 6.0, g)) + 0.05 * e * _noise((Ho, Wo), g)).contiguous()
    rms = probe.abs().square().mean().sqrt()
    probe = (probe * torch.exp(0.2j * e * _smooth((N, N), N / 10, g)) + 0.02 * e * rms * _noise((K, N, N), g)).contiguous()
    return dict(case=case, obj=obj, probe=probe, iobs=iobs, positions=pos, mask=mask, h=h,
                background=None if bg is None else (0.7 * bg).contiguous(), generator=g)


def _exit_waves(s, spread):
    """Exit waves as the previous cycle left them: P O with a relative difference of `spread`."""
    case = s["case"]
    psi = torch.empty((case["J"], case["K"], case["N"], case["N"]), dtype=torch.complex64, device="cuda")
    for lo, hi in _chunks(case):
        w = _patches(s["obj"], s["positions"], case["N"], lo, hi)[:, None] * s["probe"]
        psi[lo:hi] = w * (1 + spread * _noise(tuple(w.shape), s["generator"]))
    return psi


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fft":
        g = torch.Generator(device="cuda").manual_seed(seed)
        return dict(case=case, x=_noise((case["J"], case["N"], case["N"]), g))
    if kind == "batch":
        parts = [_scan(c, seed * 100 + i) for i, c in enumerate(_problems(case))]
        for s in parts:
            s["psi"] = _exit_waves(s, 0.1)
        pb = PtychoBatch([{k: s[k] for k in ("obj", "probe", "iobs", "positions", "mask", "psi")} for s in parts])
        return dict(case=case, pb=pb, parts=parts, algorithms=[s["case"]["kind"].upper() for s in parts])
    s = _scan(case, seed)
    psi = _exit_waves(s, 0.03 if kind == "pos" else 0.1) if kind in ("ap", "dm", "pos") else None
    pb = Ptycho(s["obj"], s["probe"], s["iobs"], s["positions"], s["mask"], psi=psi, with_psi=psi is not None,
                nearfield=case.get("nearfield") or 0.0, background=s["background"])
    return dict(case=case, pb=pb)


def run(state):
    """One call as a reconstruction program makes it, and everything it
    updates.  The likelihood is a sum of terms of single precision and is
    taken down as one."""
    case = state["case"]
    kind = case["kind"]
    if kind == "fft":
        return fft2(state["x"], case["direction"])
    pb = state["pb"]
    if kind == "batch":
        llk = pb.cycles(case["cycles"], state["algorithms"])
        return dict(llk=llk.float(), scans=[dict(obj=s["obj"], probe=s["probe"], psi=s["psi"]) for s in state["parts"]])
    if kind == "ap":
        bg = pb.background is not None
        llk = pb.ap(case["cycles"], update_background=bg)
        out = dict(obj=pb.obj, probe=pb.probe, psi=pb.psi, llk=llk.float())
        if bg:
            out["background"] = pb.background
        return out
    if kind == "dm":
        llk = pb.dm(case["cycles"])
        return dict(obj=pb.obj, probe=pb.probe, psi=pb.psi, llk=llk.float())
    if kind == "grad":
        llk, go, gp = pb.ml_grad()
        return dict(grad_obj=go, grad_probe=gp, llk=llk.float())
    if kind == "cg":
        llk = pb.ml(case["cycles"], update_obj=True, update_probe=case["update_probe"], restart=True)
        return dict(obj=pb.obj, probe=pb.probe, llk=llk.float())
    if kind == "llk":
        return pb.llk().float()
    return pb.position_shifts()


def work(case):
    """Each input read once and each output written once; 5 N log2 N
    operations per line transform and the element-wise steps."""
    kind = case["kind"]
    if kind == "fft":
        px = case["J"] * case["N"] ** 2
        return dict(bytes=16.0 * px, flops=10.0 * px * math.log2(case["N"]))
    b = f = 0.0
    for c in _problems(case):
        N, K, J = c["N"], c["K"], c["J"]
        px = float(J) * N * N
        op = 8.0 * (c["Ho"] * c["Wo"] + K * N * N)  # object and probe once
        fft = 10.0 * math.log2(N) * K * px  # one 2D transform of every wave
        if kind == "batch" or kind in ("ap", "dm"):
            near = 2 if c.get("nearfield") else 1
            dm = c["kind"] == "dm"
            b += c["cycles"] * ((16.0 if dm else 8.0) * K * px + 4.0 * px + 2 * op)
            f += c["cycles"] * (2 * near * fft + px * (K * (34.0 + (4 if dm else 0)) + 30.0))
        elif kind == "grad":
            b += 4.0 * px + 2 * op
            f += 2 * fft + px * (30.0 * K + 30.0)
        elif kind == "cg":
            waves = 3 if c["update_probe"] else 2
            b += c["cycles"] * (4.0 * px + 2 * op)
            f += c["cycles"] * ((2 + waves) * fft + px * (60.0 * K + 60.0))
        elif kind == "llk":
            b += 4.0 * px + op
            f += fft + px * (10.0 * K + 25.0)
        else:  # position shifts
            b += 8.0 * K * px + op + 8.0 * J
            f += 60.0 * K * px
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- 64-bit results


class _Exact:
    """One scan in 64 bits, by the definitions of the operators."""

    def __init__(self, s, psi=None):
        self.case = s["case"]
        self.N, self.K, self.J = (self.case[k] for k in ("N", "K", "J"))
        self.O, self.P = s["obj"].to(torch.complex128), s["probe"].to(torch.complex128)
        self.psi = None if psi is None else psi.to(torch.complex128)
        self.iobs, self.pos = s["iobs"], s["positions"]
        self.good = None if s["mask"] is None else torch.as_tensor(s["mask"], device="cuda") == 0
        self.h = _transfer(self.case, torch.complex128)
        self.bg = None if s["background"] is None else s["background"].to(torch.float64)

    def waves(self, lo, hi, O=None, P=None):
        O = self.O if O is None else O
        P = self.P if P is None else P
        return _patches(O, self.pos, self.N, lo, hi)[:, None] * P

    def model(self, F):
        ic = F.abs().square().sum(1)
        return ic if self.bg is None else ic + self.bg

    def keep(self, v):
        return v if self.good is None else torch.where(self.good, v, torch.zeros((), dtype=v.dtype, device=v.device))

    def llk_of(self, ic, io):
        return self.keep(ic - io + torch.xlogy(io, io / ic)).sum()

    def add_patches(self, acc, lo, values):
        N = self.N
        for i, (r, c) in enumerate(self.pos[lo:lo + values.shape[0]].tolist()):
            acc[r:r + N, c:c + N] += values[i]

    def cycle(self, dm, update_background):
        total = torch.zeros((), dtype=torch.float64, device="cuda")
        bsum = None if self.bg is None else torch.zeros_like(self.bg)
        np_, dp = torch.zeros_like(self.P), torch.zeros((self.N, self.N), dtype=torch.float64, device="cuda")
        for lo, hi in _chunks(self.case, 1 << 24):
            phi = self.waves(lo, hi)
            F = _detect(2 * phi - self.psi[lo:hi] if dm else phi, self.h)
            io, ic = self.iobs[lo:hi].double(), self.model(F)
            total += self.llk_of(ic, io)
            if bsum is not None:
                bsum += self.keep(io / ic).sum(0)
            self.psi[lo:hi] = phi + _undetect(self.keep((io / ic).sqrt() - 1)[:, None] * F, self.h)
            o = _patches(self.O, self.pos, self.N, lo, hi)
            np_ += (o.conj()[:, None] * self.psi[lo:hi]).sum(0)
            dp += o.abs().square().sum(0)
        if bsum is not None and update_background:
            new = self.bg * bsum / self.J
            self.bg = new if self.good is None else torch.where(self.good, new, self.bg)
        d = 0.01 * dp.max()
        self.P = (np_ + d * self.P) / (dp + d)
        no, do = torch.zeros_like(self.O), torch.zeros(self.O.shape, dtype=torch.float64, device="cuda")
        p2 = self.P.abs().square().sum(0)
        for lo, hi in _chunks(self.case, 1 << 24):
            self.add_patches(no, lo, (self.P.conj() * self.psi[lo:hi]).sum(1))
            self.add_patches(do, lo, p2.expand(hi - lo, -1, -1))
        d = 0.01 * do.max()
        self.O = (no + d * self.O) / (do + d)
        return total

    def grad(self):
        total = torch.zeros((), dtype=torch.float64, device="cuda")
        go, gp = torch.zeros_like(self.O), torch.zeros_like(self.P)
        for lo, hi in _chunks(self.case, 1 << 24):
            F = _detect(self.waves(lo, hi), None)
            io, ic = self.iobs[lo:hi].double(), self.model(F)
            total += self.llk_of(ic, io)
            w = _undetect(self.keep(2 * (1 - io / ic))[:, None] * F, None)
            self.add_patches(go, lo, (self.P.conj() * w).sum(1))
            gp += (_patches(self.O, self.pos, self.N, lo, hi).conj()[:, None] * w).sum(0)
        return total, go, gp

    def line(self, do, dp):
        l1 = torch.zeros((), dtype=torch.float64, device="cuda")
        l2 = l1.clone()
        for lo, hi in _chunks(self.case, 1 << 23):
            A = _detect(self.waves(lo, hi), None)
            B = _detect(self.waves(lo, hi, O=do) + self.waves(lo, hi, P=dp), None)
            C = _detect(self.waves(lo, hi, O=do, P=dp), None)
            io, ic = self.iobs[lo:hi].double(), self.model(A)
            di = 2 * (A.conj() * B).real.sum(1)
            d2 = 2 * (B.abs().square() + 2 * (A.conj() * C).real).sum(1)
            l1 += self.keep((1 - io / ic) * di).sum()
            l2 += self.keep((1 - io / ic) * d2 + io * (di / ic) ** 2).sum()
        return l1, l2

    def shifts(self, filter_ratio=0.1):
        O, (Ho, Wo) = self.O, self.O.shape

        def slope(v, n):  # central differences along the first axis, one-sided on its edges
            i = torch.arange(n, device=v.device)
            a, b = (i - 1).clamp_min(0), (i + 1).clamp_max(n - 1)
            return (v[b] - v[a]) / (b - a)[:, None]

        gy, gx = slope(O, Ho), slope(O.T, Wo).T
        sums = []
        for lo, hi in _chunks(self.case, 1 << 24):
            chi = self.psi[lo:hi] - self.waves(lo, hi)
            a, b = self.waves(lo, hi, O=gy), self.waves(lo, hi, O=gx)
            sums.append(torch.stack([(u.conj() * v).real.sum((1, 2, 3)) for u, v in ((a, a), (a, b), (b, b), (a, chi), (b, chi))]))
        yy, yx, xx, yc, xc = torch.cat(sums, 1)
        det, norm = yy * xx - yx * yx, yy + xx
        ok = (norm >= filter_ratio * norm.mean()) & (det > 1e-12 * norm * norm)
        z = torch.zeros_like(det)
        return torch.stack([torch.where(ok, (xx * yc - yx * xc) / det, z), torch.where(ok, (yy * xc - yx * yc) / det, z)], 1)


def _dot(a, b):
    return sum((u.conj() * v).real.sum() for u, v in zip(a, b))


def exact(case, seed):
    kind = case["kind"]
    if kind == "fft":
        f = torch.fft.fft2 if case["direction"] < 0 else torch.fft.ifft2
        x = prepare(case, seed)["x"].to(torch.complex128)
        for i in range(0, x.shape[0], 256):
            x[i:i + 256] = f(x[i:i + 256], norm="ortho")
        return x
    if kind == "batch":
        llks, scans = [], []
        for i, c in enumerate(_problems(case)):
            s = _scan(c, seed * 100 + i)
            e = _Exact(s, _exit_waves(s, 0.1))
            llks.append(torch.stack([e.cycle(c["kind"] == "dm", False) for _ in range(case["cycles"])]))
            scans.append(dict(obj=e.O, probe=e.P, psi=e.psi))
        return dict(llk=torch.stack(llks, 1), scans=scans)
    s = _scan(case, seed)
    psi = _exit_waves(s, 0.03 if kind == "pos" else 0.1) if kind in ("ap", "dm", "pos") else None
    e = _Exact(s, psi)
    del psi
    if kind in ("ap", "dm"):
        llk = torch.stack([e.cycle(kind == "dm", e.bg is not None) for _ in range(case["cycles"])])
        out = dict(obj=e.O, probe=e.P, psi=e.psi, llk=llk)
        if e.bg is not None:
            out["background"] = e.bg
        return out
    if kind == "grad":
        llk, go, gp = e.grad()
        return dict(grad_obj=go, grad_probe=gp, llk=llk)
    if kind == "cg":
        llks, prev, d = [], None, None
        for _ in range(case["cycles"]):
            llk, go, gp = e.grad()
            gp = gp if case["update_probe"] else torch.zeros_like(gp)
            beta = 0.0
            if prev is not None:
                beta = max(0.0, float((_dot((go, gp), (go, gp)) - _dot((go, gp), prev)) / _dot(prev, prev)))
            d = (-go, -gp) if d is None else (-go + beta * d[0], -gp + beta * d[1])
            prev = (go, gp)
            l1, l2 = e.line(*d)
            alpha = float(-l1 / l2) if float(l2) > 0 else 0.0
            e.O, e.P = e.O + alpha * d[0], e.P + alpha * d[1]
            llks.append(llk)
        return dict(obj=e.O, probe=e.P, llk=torch.stack(llks))
    if kind == "llk":
        return sum(e.llk_of(e.model(F), e.iobs[lo:hi].double())
                   for lo, hi in _chunks(case, 1 << 24) for F in (_detect(e.waves(lo, hi), None),))
    return e.shifts()
