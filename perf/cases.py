"""The calls that this library's speed is measured on, and what they give in 64 bits.

Every case is one pass through the public entry points of ``paper_2204_08269_gb300`` as a user's
program makes it: a batched or single forward transform, a fused forward + backward step, the
autograd module under a loss, the uneven-length graph, the Eq. 5 similarity features, time
scattering, and the end-to-end step on host buffers.  Parameters are the repository's own
benchmark and test configurations.

``exact`` recomputes the outputs with plain torch operations in float64 (FFTs, dense products,
torch's own autograd for the gradients), from the formulas of the filterbanks and the
subsampling schedule; it uses none of the library's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2204_08269_gb300 import JTFS, JTFSPlan
from paper_2204_08269_gb300 import jtfs as lib
from paper_2204_08269_gb300.resynth import normalised_error

SR = 22050.0

# parameter families: the batched benchmark, its mixed-precision form, the plain single
# transform, the 32-frame test configuration, texture resynthesis, the Eq. 5 similarity study
# and the time-scattering comparison
AUDIO = dict(J=12, Q=16, J_fr=4, Q_fr=2, T=2 ** 12, F=16)
MIXED = dict(J=11, Q=12, J_fr=4, Q_fr=1, T=2 ** 11, F=12)
PLAIN = dict(J=6, Q=8, J_fr=3, Q_fr=1, T=2 ** 6, F=8)
FRAMES32 = dict(J=8, Q=16, J_fr=3, Q_fr=2, T=2 ** 8, F=16)
TEXTURE = dict(J=13, Q=16, J_fr=4, Q_fr=2, T=2 ** 13, F=16)
STUDY = dict(J=14, Q=8, J_fr=4, Q_fr=1, T=2 ** 14, F=1)
SCAT1D = dict(J=13, Q=16, J_fr=4, Q_fr=1, T=2 ** 11, F=4)


def _case(name, kind, family, N, B, precision="fp32", **more):
    c = dict(kind=kind, N=N, B=B, precision=precision, **family, **more)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # one short signal, forward only: the latency of a single small transform
        _case("forward_1x4096", "forward", PLAIN, 2 ** 12, 1, signal="chirp"),
        # one three-second signal, value and gradient: the paper's own setting (a single sound
        # optimised by gradient descent), where one signal has to fill the GPU
        _case("step_1x65536", "step", AUDIO, 2 ** 16, 1, signal="amfm"),
        # the headline: 64 signals, value and gradient in one call
        _case("step_64x65536", "step", AUDIO, 2 ** 16, 64, signal="amfm"),
        # a small odd batch in BF16, value and gradient
        _case("step_5x65536_bf16", "step", AUDIO, 2 ** 16, 5, "bf16", signal="amfm"),
        # feature extraction for a dataset: the largest batch, forward only, BF16 contraction
        _case("forward_256x32768_bf16", "forward", MIXED, 2 ** 15, 256, "bf16", signal="amfm"),
        # the same with the TF32 contraction, on a batch that is no round number
        _case("forward_77x32768_tf32", "forward", MIXED, 2 ** 15, 77, "tf32", signal="amfm"),
        # texture resynthesis: the autograd module under the normalised-error loss
        _case("texture_16x131072", "texture", TEXTURE, 2 ** 17, 16, signal="clicks"),
        # a dataset of recordings of different lengths, value and gradient, one graph replay
        _case("uneven_96", "uneven", AUDIO, 2 ** 17, 96, length_seed=20220413, chunk=64),
        # similarity study: Eq. 4 (no frequential averaging) and mu-log features of 64 chirps
        _case("study_64x65536", "study", STUDY, 2 ** 16, 64, signal="eq5", average_fr=False),
        # the time-scattering baseline, value and gradient
        _case("scattering1d_32x65536", "scat1d", SCAT1D, 2 ** 16, 32, signal="amfm"),
        # every second-order path (the phi_t paths too) in the single 2-D output layout
        _case("all_paths_33x8192", "step", FRAMES32, 2 ** 13, 33, signal="amfm", branches=15,
              out_3d=False),
        # end to end from pinned host buffers: copies in and out inside the call
        _case("host_step_32x65536", "host", AUDIO, 2 ** 16, 32, signal="amfm"),
    ]


def draw(rng):
    """One more case: the kinds, families, precisions and sizes of the listed ones, batches
    log-uniform up to the number that makes the listed case of that kind."""
    def batch(most):
        return max(1, min(most, int(round(math.exp(rng.uniform(0.0, math.log(most + 0.49)))))))

    kind = rng.choice(["forward", "forward", "step", "step", "texture", "uneven", "study",
                       "scat1d", "host"])
    if kind in ("forward", "step", "host"):
        family, lengths = rng.choice([(AUDIO, (15, 16, 17)), (MIXED, (13, 14, 15)),
                                      (PLAIN, (9, 10, 11, 12)), (FRAMES32, (11, 12, 13))])
        logn = rng.choice(lengths)
        precisions = ["fp32", "fp32", "bf16"]
        if kind != "step" and (1 << logn) // family["T"] <= 16:
            precisions.append("tf32")
        more = {}
        if kind != "host" and rng.random() < 0.3:
            more = dict(branches=15, out_3d=rng.random() < 0.5)
        most = {"forward": 2 ** 22, "step": 2 ** 21, "host": 2 ** 20}[kind] >> logn
        return _case(None, kind, family, 1 << logn, batch(min(256, most)), rng.choice(precisions),
                     signal=rng.choice(["amfm", "clicks"]), **more)
    if kind == "texture":
        family, logn = rng.choice([(TEXTURE, 16), (TEXTURE, 17), (AUDIO, 16), (MIXED, 15)])
        return _case(None, kind, family, 1 << logn, batch(2 ** 20 >> logn),
                     rng.choice(["fp32", "fp32", "bf16"]), signal="clicks")
    if kind == "uneven":
        return _case(None, kind, AUDIO, 2 ** 17, batch(64), rng.choice(["fp32", "fp32", "bf16"]),
                     length_seed=rng.randrange(1 << 30), chunk=rng.choice([16, 32, 64]))
    if kind == "study":
        return _case(None, kind, STUDY, 2 ** 16, batch(64), signal="eq5", average_fr=False)
    logn = rng.choice([14, 15, 16])
    return _case(None, kind, rng.choice([SCAT1D, MIXED]), 1 << logn, batch(2 ** 20 >> logn),
                 signal="amfm")


# ----------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------
def _uniform(rng, lo, hi, n):
    return torch.from_numpy(rng.uniform(lo, hi, size=(n, 1))).cuda()


def _amfm(B, N, rng):
    """AM/FM tones with white noise 30 dB down: carrier log-uniform in 100-4000 Hz, AM 1-16 Hz
    (depth 0.5), FM 1-8 Hz with an excursion of 1-6 semitones."""
    t = torch.arange(N, dtype=torch.float64, device="cuda") / SR
    fc = torch.exp(_uniform(rng, math.log(100.0), math.log(4000.0), B))
    fam, ffm, e = _uniform(rng, 1, 16, B), _uniform(rng, 1, 8, B), _uniform(rng, 1, 6, B)
    p1, p2 = _uniform(rng, 0, 2 * math.pi, B), _uniform(rng, 0, 2 * math.pi, B)
    inst = fc * 2.0 ** ((e / 12.0) * torch.sin(2 * math.pi * ffm * t + p2))
    phi = 2 * math.pi * torch.cumsum(inst, dim=1) / SR
    tone = (1 + 0.5 * torch.sin(2 * math.pi * fam * t + p1)) * torch.sin(phi)
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    noise = torch.randn(tone.shape, dtype=torch.float64, device="cuda", generator=gen)
    return (tone + noise * tone.square().mean(dim=1, keepdim=True).sqrt() * 10 ** -1.5).float()


def _clicks(B, N, rng):
    """Poisson click trains (5-40 Hz), every click through its own second-order resonator
    (200-6000 Hz, Q log-uniform in 5-30), unit RMS, white noise 40 dB down."""
    out = torch.empty((B, N), dtype=torch.float32, device="cuda")
    w = 2 * math.pi * torch.arange(N // 2 + 1, dtype=torch.float64, device="cuda") / N
    z1 = torch.polar(torch.ones_like(w), -w)
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    for b in range(B):
        n = max(1, int(rng.poisson(rng.uniform(5.0, 40.0) * N / SR)))
        w0 = 2 * math.pi * _uniform(rng, 200, 6000, n) / SR
        alpha = torch.sin(w0) / (2 * torch.exp(_uniform(rng, math.log(5.0), math.log(30.0), n)))
        amp = _uniform(rng, 0.5, 1.0, n) * torch.from_numpy(
            np.where(rng.random((n, 1)) < 0.5, 1.0, -1.0)).cuda()
        pos = torch.from_numpy(rng.integers(0, N, size=(n, 1)).astype(np.float64)).cuda()
        spec = torch.zeros_like(z1)
        for i in range(0, n, 32):
            j = slice(i, i + 32)
            h = alpha[j] * (1 - z1 * z1) / (
                (1 + alpha[j]) - 2 * torch.cos(w0[j]) * z1 + (1 - alpha[j]) * z1 * z1)
            spec = spec + (amp[j] * h * torch.polar(torch.ones_like(h.real), -w * pos[j])).sum(0)
        y = torch.fft.irfft(spec, n=N)
        y = y / y.square().mean().sqrt().clamp_min(1e-30)
        noise = torch.randn(N, dtype=torch.float64, device="cuda", generator=gen)
        out[b] = (y + 0.01 * noise).float()
    return out


def _chirp(B, N, rng):
    """Unit white noise plus a linear chirp from 0.01 to 0.4 cycles per sample."""
    n = torch.arange(N, dtype=torch.float64, device="cuda")
    phase = 2 * math.pi * (0.01 * n + 0.39 * n * n / (2.0 * N))
    x = torch.from_numpy(rng.standard_normal((B, N))).cuda()
    return (x + 0.5 * torch.sin(phase)).float()


def _eq5(B, N, rng):
    """The paper's AM/FM exponential chirps (Sec. 3.2, Eq. 5), a window of two octaves."""
    t = (torch.arange(N, dtype=torch.float64, device="cuda") - N / 2) / SR
    fc = torch.exp(_uniform(rng, math.log(512.0), math.log(1024.0), B))
    fm = torch.exp(_uniform(rng, math.log(4.0), math.log(32.0), B))
    gm = torch.exp(_uniform(rng, math.log(0.5), math.log(4.0), B))
    return (torch.exp(-0.5 * (gm * t) ** 2) * torch.sin(2 * math.pi * fm * t) * torch.sin(
        2 * math.pi * fc / (gm * math.log(2.0)) * 2.0 ** (gm * t))).float()


SIGNALS = {"amfm": _amfm, "clicks": _clicks, "chirp": _chirp, "eq5": _eq5}


def _lengths(case):
    """Signal lengths log-uniform in 2^13 .. 2^17 (a property of the case, not of the seed)."""
    rng = np.random.default_rng(case["length_seed"])
    return np.floor(2.0 ** rng.uniform(13.0, 17.0, size=case["B"])).astype(np.int64)


def _inputs(case, seed):
    """x (or the packed uneven signals), the cotangents and, for the texture case, the target."""
    c, rng = case, np.random.default_rng(seed)
    if c["kind"] == "uneven":
        x = torch.cat([SIGNALS["amfm" if i % 2 == 0 else "clicks"](1, int(n), rng)[0]
                       for i, n in enumerate(_lengths(c))])
        return x, None
    if c["kind"] == "texture":
        target = SIGNALS[c["signal"]](c["B"], c["N"], rng)
        noise = torch.from_numpy(rng.standard_normal(target.shape).astype(np.float32)).cuda()
        return noise, target
    return SIGNALS[c["signal"]](c["B"], c["N"], rng), None


def _cotangents(sizes, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    return [torch.randn(s, device="cuda", generator=gen) for s in sizes]


def _plan_args(case):
    keys = ("N", "J", "Q", "J_fr", "Q_fr", "T", "F", "precision", "average_fr", "branches",
            "out_3d")
    return {k: case[k] for k in keys if k in case}


def prepare(case, seed):
    c = case
    x, target = _inputs(c, seed)
    st = dict(kind=c["kind"], x=x)
    if c["kind"] == "uneven":
        args = {k: v for k, v in _plan_args(c).items() if k != "N"}
        v = lib.JTFSVarlen(_lengths(c), chunk=c["chunk"], **args)
        g = _cotangents([int(o[-1]) for o in (v.s0_off, v.s1_off, v.s2_off)], seed)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            outs = v.capture(x, g)
        torch.cuda.current_stream().wait_stream(side)
        return dict(st, v=v, outs=outs, g=g)
    if c["kind"] == "texture":
        st["model"] = JTFS(**_plan_args(c))
        with torch.no_grad():
            st["goal"] = _flat(*st["model"](target))
        x.requires_grad_(True)
        return st
    plan = JTFSPlan(**_plan_args(c))
    st["plan"] = plan
    sh, B = plan.shapes, c["B"]
    if c["kind"] == "scat1d":
        st["g"] = _cotangents([sh.s0(B), sh.s1(B), (B, sh.n2, sh.n1, sh.n_t)], seed)
    elif c["kind"] in ("step", "host"):
        two = c.get("out_3d", True) is False
        st["g"] = _cotangents([sh.out_2d(B)] if two else [sh.s0(B), sh.s1(B), sh.s2(B)], seed)
    if c["kind"] == "host":
        st["x"] = x.cpu().pin_memory()
        st["g"] = [g.cpu().pin_memory() for g in st["g"]]
    return st


def _flat(s0, s1, s2):
    B = s0.shape[0]
    return torch.cat([s0.reshape(B, -1), s1.reshape(B, -1), s2.reshape(B, -1)], dim=1)


def run(state):
    s = state
    kind = s["kind"]
    if kind == "forward":
        return list(s["plan"].forward(s["x"], keep_checkpoint=False)[:3])
    if kind == "step":
        return list(s["plan"].forward_backward(s["x"], *s["g"]))
    if kind == "host":
        return list(s["plan"].forward_backward_host(s["x"], *s["g"]))
    if kind == "uneven":
        s["v"].replay()
        return s["outs"]
    if kind == "texture":
        out = s["model"](s["x"])
        loss = normalised_error(_flat(*out), s["goal"])
        (g,) = torch.autograd.grad(loss.sum(), s["x"])
        return [t.detach() for t in out] + [loss.detach(), g]
    if kind == "study":
        s0, s1, s2, _ = s["plan"].forward(s["x"], keep_checkpoint=False)
        B, n1 = s1.shape[0], s1.shape[1]
        paths = s2.reshape(B, -1, s2.shape[-2] * s2.shape[-1])
        mu = lib.mulog_mean(paths)
        return [s0, s1, s2, mu, lib.mulog(paths, mu, eps=0.1)]
    s0, s1, s2t, u1 = s["plan"].scattering1d(s["x"])
    return [s0, s1, s2t, s["plan"].scattering1d_backward(s["x"], u1, *s["g"])]


# ----------------------------------------------------------------------------------------
# the transform in 64 bits
# ----------------------------------------------------------------------------------------
FWHM = 2.0 * math.sqrt(2.0 * math.log(2.0))


def _bank(J, Q):
    rho = (1.0 - 2.0 ** (-1.0 / Q)) / FWHM
    top, least = min(0.35, 0.5 / (1.0 + 4.0 * rho)), 0.1 * 2.0 ** -J
    xi, sg = [], []
    while rho * top * 2.0 ** (-len(xi) / Q) >= least:
        xi.append(top * 2.0 ** (-len(xi) / Q))
        sg.append(rho * xi[-1])
    last = xi[-1]
    m = 1
    while last - m * FWHM * least >= FWHM * least:
        xi.append(last - m * FWHM * least)
        sg.append(least)
        m += 1
    return np.array(xi), np.array(sg)


def _morlet(w, xi, sg):
    v = np.exp(-(w - xi) ** 2 / (2 * sg * sg)) - math.exp(-xi * xi / (2 * sg * sg)) * np.exp(
        -w * w / (2 * sg * sg))
    return np.where((w > 0) & (w < 0.5), v, 0.0)


def _filters(xi, sg, low, G, w):
    """The bank on the frequencies w, scaled so that its Littlewood-Paley sum on the G-point
    grid stays at or below one."""
    om = np.arange(1, G // 2) / G
    p = np.zeros_like(om)
    for a, b in zip(xi, sg):
        p += 0.5 * _morlet(om, a, b) ** 2
    ok = p > 0
    c = math.sqrt(float(np.min((1 - np.exp(-om * om / (low * low)))[ok] / p[ok])))
    return [c * _morlet(w, a, b) for a, b in zip(xi, sg)]


class Exact:
    """Filters and schedule of one configuration in float64 on the GPU."""

    def __init__(self, case, N=None):
        c = case
        N = self.N = N or c["N"]
        T, F = c["T"], c["F"]
        self.T, self.n_t = T, N // T
        xi1, sg1 = (v[::-1].copy() for v in _bank(c["J"], c["Q"]))
        xi2, sg2 = _bank(c["J"], 1)
        xif, sgf = _bank(c["J_fr"], c["Q_fr"])
        n1 = self.n1 = len(xi1)
        self.n2, self.n_fr = len(xi2), len(xif)
        self.C = 2 * self.n_fr + 1
        Nf = 2 * (1 << math.ceil(math.log2(n1)))
        self.avg = c.get("average_fr", True)
        stride = 1 << int(math.floor(math.log2(F)))
        self.n_lo = -(-n1 // stride) if self.avg else n1
        w = np.arange(N // 2) / N

        def dev(v):
            return torch.from_numpy(np.ascontiguousarray(v)).cuda()

        self.psi1 = dev(np.stack(_filters(xi1, sg1, 0.1 / T, N, w)))
        self.psi2 = dev(np.stack(_filters(xi2, sg2, 0.1 / T, N, w)))
        full = np.fft.fftfreq(N)
        self.phiT = dev(np.fft.ifft(np.exp(-full ** 2 / (2 * (0.1 / T) ** 2))).real)
        wf = np.fft.fftfreq(Nf)
        wf[Nf // 2] = 0.5
        up = np.stack(_filters(xif, sgf, 0.1 / F, Nf, wf))
        down = np.stack(_filters(xif, sgf, 0.1 / F, Nf, -wf))
        phiF = np.exp(-wf ** 2 / (2 * (0.1 / F) ** 2))
        h = np.fft.ifft(np.concatenate([up, down, phiF[None]]), axis=-1)
        lam = np.arange(n1)
        self.W = dev(h[:, (lam[:, None] - lam[None, :]) % Nf])
        lo = np.arange(self.n_lo)
        self.PhiF = dev(np.fft.ifft(phiF).real[(lo[:, None] * stride - lam[None, :]) % Nf])
        br = c.get("branches", 3) or 3
        self.phi_c = (list(range(self.n_fr)) if br & 4 else []) + (
            [2 * self.n_fr] if br & 8 else [])

        def pow2(v):
            return min(T, 1 << max(0, math.floor(math.log2(v))))

        self.s1 = [pow2(1.0 / (16.0 * s)) for s in sg1]
        nyq = 0.5 / min(self.s1)
        self.rates = []
        for a in range(self.n2):
            lo_, hi = max(0.0, xi2[a] - 4 * sg2[a]), min(xi2[a] + 4 * sg2[a], nyq)
            if lo_ >= hi:
                self.rates.append(None)
                continue
            keep = [l for l in range(n1) if 0.5 / self.s1[l] > lo_]
            self.rates.append((pow2(1.0 / (2.0 * (hi - lo_))), keep[0] if keep else n1))
        self._pool = {}
        # rows of one stride are consecutive: [first, end)
        self.groups = []
        for l in range(n1):
            if self.groups and self.s1[self.groups[-1][0]] == self.s1[l]:
                self.groups[-1][1] = l + 1
            else:
                self.groups.append([l, l + 1])

    def pool(self, u, s):
        """Riemann sum of phi_T at stride s, every T samples."""
        if s not in self._pool:
            t = torch.arange(self.n_t, device="cuda")[:, None] * self.T
            m = torch.arange(self.N // s, device="cuda")[None, :] * s
            self._pool[s] = (s * self.phiT[(t - m) % self.N]).T.contiguous()
        return u @ self._pool[s]

    @staticmethod
    def _fold(P, L):
        """The bins of P (last axis, from bin 0) summed modulo L."""
        n = P.shape[-1]
        if n % L:
            P = torch.nn.functional.pad(P, (0, L - n % L))
        return P.reshape(P.shape[:-1] + (-1, L)).sum(dim=-2)

    def first(self, x):
        """S0, S1 and the scalogram rows by group of x [B, N] (float64)."""
        xh = torch.fft.fft(x)[:, None, :self.N // 2]
        U, S1 = [], []
        for l0, l1 in self.groups:
            s = self.s1[l0]
            L = self.N // s
            z = torch.fft.ifft(self._fold(xh * self.psi1[l0:l1], L)) * (L / self.N)
            U.append(z.abs())
            S1.append(self.pool(U[-1], s))
        return self.pool(x, 1), torch.cat(S1, dim=1), U

    def rows(self, U, a):
        """Y_alpha [B, n1 - lam_min, L_alpha]."""
        s, lm = self.rates[a]
        La = self.N // s
        out = []
        for (l0, l1), u in zip(self.groups, U):
            l = max(l0, lm)
            if l >= l1:
                continue
            Lr = u.shape[-1]
            Uh = torch.fft.fft(u[:, l - l0:])[..., :Lr // 2] * self.psi2[a, :Lr // 2]
            out.append(torch.fft.ifft(self._fold(Uh, La)) * (La / Lr))
        return torch.cat(out, dim=1)

    def modulus_paths(self, W, Y, s):
        """phi_F phi_T |W Y| of Y [B, K, L] for W [C, n1, K]."""
        C, n1, K = W.shape
        Z = (W.reshape(C * n1, K) @ Y).reshape(Y.shape[0], C, n1, -1)
        P = self.pool(Z.abs(), s)
        return self.PhiF @ P if self.avg else P

    def joint(self, x):
        S0, S1, U = self.first(x)
        S2 = []
        for a, r in enumerate(self.rates):
            if r is None or r[1] >= self.n1:
                S2.append(x.new_zeros((x.shape[0], self.C, self.n_lo, self.n_t)))
            else:
                S2.append(self.modulus_paths(self.W[:, :, r[1]:], self.rows(U, a), r[0]))
        S2 = torch.stack(S2, dim=1)
        if self.phi_c:
            tail = self.modulus_paths(self.W[self.phi_c], S1.to(torch.complex128), self.T)
            S2 = torch.cat([S2.flatten(1, 2), tail], dim=1)
        return S0, S1, S2

    def time(self, x):
        S0, S1, U = self.first(x)
        S2 = []
        for a, r in enumerate(self.rates):
            full = x.new_zeros((x.shape[0], self.n1, self.n_t))
            if r is not None and r[1] < self.n1:
                P = self.pool(self.rows(U, a).abs(), r[0])
                full = torch.cat([full[:, :r[1]], P], dim=1)
            S2.append(full)
        return S0, S1, torch.stack(S2, dim=1)


def _by_signals(f, B, at_once):
    parts = [f(slice(i, min(B, i + at_once))) for i in range(0, B, at_once)]
    return [torch.cat(p) for p in zip(*parts)]


def _at_once(case):
    return max(1, min(16, 2 ** 19 // case["N"]))


def _exact_uneven(case, x, g):
    n = [int(v) for v in _lengths(case)]
    pad = [max(1 << max(0, v - 1).bit_length(), 1 << (case["J"] + 3)) for v in n]
    frames = [-(-v // case["T"]) for v in n]
    models = {N: Exact(case, N) for N in sorted(set(pad))}
    paths = [[1, E.n1, E.n2 * E.C * E.n_lo] for E in (models[p] for p in pad)]
    off = np.cumsum([[0] * 3] + [[r * f for r in rows] for rows, f in zip(paths, frames)], axis=0)
    xo = np.concatenate([[0], np.cumsum(n)])
    outs = [torch.empty(int(off[-1][k]), dtype=torch.float64, device="cuda") for k in range(3)]
    gx = torch.empty(int(xo[-1]), dtype=torch.float64, device="cuda")
    for i, N in enumerate(pad):
        xi = torch.zeros((1, N), dtype=torch.float64, device="cuda")
        xi[0, :n[i]] = x[xo[i]:xo[i + 1]].double()
        xi.requires_grad_(True)
        total = 0.0
        for k, s in enumerate(models[N].joint(xi)):
            s = s.reshape(paths[i][k], -1)[:, :frames[i]].reshape(-1)
            where = slice(int(off[i][k]), int(off[i + 1][k]))
            outs[k][where] = s.detach()
            total = total + (s * g[k][where].double()).sum()
        gx[xo[i]:xo[i + 1]] = torch.autograd.grad(total, xi)[0][0, :n[i]]
    return outs + [gx]


def exact(case, seed):
    c = case
    x, target = _inputs(c, seed)
    if c["kind"] == "uneven":
        lens = _lengths(c)
        E = {}
        total = [0, 0, 0]
        for v in lens:
            N = max(1 << max(0, int(v) - 1).bit_length(), 1 << (c["J"] + 3))
            e = E.setdefault(N, Exact(c, N))
            f = -(-int(v) // c["T"])
            for k, r in enumerate((1, e.n1, e.n2 * e.C * e.n_lo)):
                total[k] += r * f
        E.clear()
        return _exact_uneven(c, x, _cotangents(total, seed))
    E, B, two = Exact(c), c["B"], c.get("out_3d", True) is False
    forward = E.time if c["kind"] == "scat1d" else E.joint

    def outputs(v):
        S0, S1, S2 = forward(v)
        if not two:
            return [S0, S1, S2]
        rows = S2.reshape(v.shape[0], -1, E.n_t)
        return [torch.cat([S0[:, None], S1, rows], dim=1)]

    if c["kind"] in ("forward", "study"):
        with torch.no_grad():
            out = _by_signals(lambda i: outputs(x[i].double()), B, _at_once(c))
        if c["kind"] == "study":
            P = out[2].reshape(B, -1, E.n_lo * E.n_t)
            mu = P.sum(dim=2).mean(dim=0)
            out += [mu, torch.log1p(P / (0.1 * mu[:, None]))]
        return out
    if c["kind"] == "texture":
        def part(i):
            with torch.no_grad():
                goal = _flat(*E.joint(target[i].double()))
            v = x[i].double().requires_grad_(True)
            out = E.joint(v)
            loss = (_flat(*out) - goal).norm(dim=1) / goal.norm(dim=1)
            (gv,) = torch.autograd.grad(loss.sum(), v)
            return [t.detach() for t in out] + [loss.detach(), gv]
        return _by_signals(part, B, _at_once(c))
    s2 = (B, E.n2, E.n1, E.n_t) if c["kind"] == "scat1d" else (
        (B, E.n2 * E.C + len(E.phi_c), E.n_lo, E.n_t) if E.phi_c else
        (B, E.n2, E.C, E.n_lo, E.n_t))
    sizes = [(B, E.n_t), (B, E.n1, E.n_t), s2]
    if two:
        sizes = [(B, 1 + E.n1 + (E.n2 * E.C + len(E.phi_c)) * E.n_lo, E.n_t)]
    g = _cotangents(sizes, seed)

    def part(i):
        v = x[i].double().requires_grad_(True)
        out = outputs(v)
        (gv,) = torch.autograd.grad(out, v, [t[i].double() for t in g])
        return [t.detach() for t in out] + [gv]

    out = _by_signals(part, B, _at_once(c))
    if two:
        out = [out[0], None, None, out[1]]
    if c["kind"] == "host":
        out = [t.cpu() for t in out]
    return out


# ----------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------
def _sizes(case, N):
    """(values of the outputs, flops of one forward) per signal of N samples.  The spin-down
    channels follow from the spin-up products, so a forward takes 8 (n_fr + 1) n1 sum K L real
    operations for the contraction, plus the phi_T pooling and the FFTs."""
    c = case
    xi1, sg1 = _bank(c["J"], c["Q"])
    xi2, sg2 = _bank(c["J"], 1)
    n1, n2, nfr = len(xi1), len(xi2), len(_bank(c["J_fr"], c["Q_fr"])[0])
    T, n_t, C = c["T"], N // c["T"], 2 * nfr + 1
    n_lo = -(-n1 // (1 << int(math.log2(c["F"])))) if c.get("average_fr", True) else n1

    def pow2(v):
        return min(T, 1 << max(0, math.floor(math.log2(v))))

    s1 = [pow2(1.0 / (16.0 * s)) for s in sg1]
    flops = 2.5 * N * math.log2(N) + sum(7.5 * (N // s) * math.log2(max(2, N // s)) for s in s1)
    for a in range(n2):
        lo, hi = max(0.0, xi2[a] - 4 * sg2[a]), min(xi2[a] + 4 * sg2[a], 0.5 / min(s1))
        if lo >= hi:
            continue
        L = N // pow2(1.0 / (2.0 * (hi - lo)))
        K = sum(0.5 / s > lo for s in s1)
        flops += 5.0 * K * L * math.log2(max(2, L))
        if c["kind"] == "scat1d":
            flops += 2.0 * K * L * n_t
        else:
            flops += 8.0 * (nfr + 1) * n1 * K * L + 2.0 * C * n1 * L * n_t
    br = c.get("branches", 3) or 3
    paths = n2 * n1 if c["kind"] == "scat1d" else (
        n2 * C + (nfr if br & 4 else 0) + (1 if br & 8 else 0)) * n_lo
    return (1 + n1 + paths) * n_t, flops


def work(case):
    c = case
    if c["kind"] == "uneven":
        nbytes = flops = 0.0
        for n in _lengths(c):
            N = max(1 << max(0, int(n) - 1).bit_length(), 1 << (c["J"] + 3))
            values, f = _sizes(c, N)
            kept = values * -(-int(n) // c["T"]) // (N // c["T"])
            nbytes += 4.0 * (2 * int(n) + 2 * kept)
            flops += 3.0 * f
        return {"bytes": nbytes, "flops": flops}
    values, f = _sizes(c, c["N"])
    grad = c["kind"] in ("step", "host", "texture", "scat1d")
    per = (c["N"] + values) * (2 if grad else 1)
    if c["kind"] == "study":
        per += 2 * values          # mu-log reads S2 and writes its features
    return {"bytes": 4.0 * c["B"] * per, "flops": float(c["B"] * f * (3 if grad else 1))}
