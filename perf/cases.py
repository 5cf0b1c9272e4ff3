"""The workloads by which the speed of this framework is judged.

A case is one pass of what a program does with the transform: the synthesis of a
batch of spectra together with the analysis of a batch of grids (what each time
step of a pseudo-spectral code calls), or one gradient step of a loss on the
synthesised fields.  ``listed()`` names the fixed cases, ``draw()`` gives others
of the same ranges, ``prepare()`` makes the inputs and the plan that a program
holds, ``run()`` is the pass, ``work()`` the bytes and operations it cannot do
without, and ``exact()`` its outputs by the definitions in 64-bit arithmetic.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1202_6522_gb300 import SHT, UnevenBatch
from paper_1202_6522_gb300 import synthetic

# kind "scalar": synthesis of `batch` spectra and analysis of `batch` grids;
# kind "vector": the same for spheroidal/toroidal pairs; kind "grad" and
# "vector_grad": loss = |synthesis - target|^2 and its gradient; kind "uneven":
# one graph launch per direction over `batch` fields of different truncations.
# `dtype` is the data's ("f64" or "f32"), `path` the plan's choice for it
# ("cc": CUDA cores, the default of SHT; "tc": tensor cores).


def _case(name, kind, dtype, path, lmax, nlat, nphi, batch, mres=1):
    return {"name": name, "kind": kind, "dtype": dtype, "path": path, "lmax": lmax, "mmax": lmax // mres,
            "nlat": nlat, "nphi": nphi, "batch": batch, "mres": mres}


def listed():
    return [
        # a tutorial-sized field, the least the library is called with: launches and host time
        _case("f64_n31_b1", "scalar", "f64", "cc", 31, 32, 64, 1),
        # the mid-sized single field of a time-stepping code, both directions each step
        _case("f64_n255_b1", "scalar", "f64", "cc", 255, 256, 512, 1),
        # velocity fields on 16 radial shells, grid dealiased by 3/2 (mixed-radix longitudes)
        _case("f64_vector_n127_b16", "vector", "f64", "cc", 127, 192, 384, 16),
        # many shells of a scalar in plain FP64
        _case("f64_n511_b16", "scalar", "f64", "cc", 511, 512, 1024, 16),
        # the benchmark's headline: FP64 data on the tensor cores, high resolution, batched
        _case("f64_tc_n1023_b16", "scalar", "f64", "tc", 1023, 1024, 2048, 16),
        # the same path at an odd truncation with a ragged batch and a mixed-radix grid
        _case("f64_tc_n340_b5", "scalar", "f64", "tc", 340, 361, 720, 5),
        # single precision on the default path: 3-fold symmetric, dealiased, few fields
        _case("f32_n383_m3_b6", "scalar", "f32", "cc", 383, 576, 384, 6, 3),
        # single precision at the highest resolution the tests run besides N = 4095
        _case("f32_n2047_b2", "scalar", "f32", "cc", 2047, 2048, 4096, 2),
        # a learned model of winds: vector synthesis and its gradient on the default path
        _case("f32_vector_grad_n511_b8", "vector_grad", "f32", "cc", 511, 512, 1024, 8),
        # 64 radial shells of a vector field in one launch on the tensor cores
        _case("f32_tc_vector_n511_b64", "vector", "f32", "tc", 511, 512, 1024, 64),
        # differentiable high-resolution transform: loss and gradient, tensor cores
        _case("f32_tc_grad_n1023_b16", "grad", "f32", "tc", 1023, 1024, 2048, 16),
        # 96 fields of truncations 63, 127, 255 and 511 in one graph launch per direction
        _case("f32_uneven_n511_b96", "uneven", "f32", "tc", 511, 512, 1024, 96),
    ]


# Range of each family of cases: kind, dtype, path, truncations, batches, and the
# largest batch * (lmax + 1)^3 (that of the family's largest listed case).
_FAMILIES = [
    ("scalar", "f64", "cc", (31, 511), (1, 16), 16 * 512 ** 3),
    ("vector", "f64", "cc", (31, 255), (1, 16), 16 * 128 ** 3),
    ("scalar", "f64", "tc", (127, 1023), (1, 16), 16 * 1024 ** 3),
    ("scalar", "f32", "cc", (63, 2047), (1, 16), 2 * 2048 ** 3),
    ("vector_grad", "f32", "cc", (63, 511), (1, 16), 8 * 512 ** 3),
    ("vector", "f32", "tc", (63, 511), (1, 64), 64 * 512 ** 3),
    ("grad", "f32", "tc", (127, 1023), (1, 16), 16 * 1024 ** 3),
    ("uneven", "f32", "tc", (63, 511), (8, 96), 96 * 512 ** 3),
]


def _log_uniform(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def _smooth_nphi(least):
    """The smallest even 2^a 3^b 5^c that is at least `least` (and twice such a number)."""
    h = (least + 1) // 2
    while True:
        q = h
        for r in (2, 3, 5):
            while q % r == 0:
                q //= r
        if q == 1:
            return 2 * h
        h += 1


def draw(rng):
    kind, dtype, path, ls, bs, most = rng.choice(_FAMILIES)
    if kind == "uneven":
        batch = rng.randint(*bs)
        return {"kind": kind, "dtype": dtype, "path": path, "lmax": 511, "mmax": 511, "nlat": 512, "nphi": 1024,
                "batch": batch, "mres": 1}
    lmax = _log_uniform(rng, *ls)
    if rng.random() < 0.5:          # half of the truncations are of the usual form 2^k - 1
        lmax = min(ls[1], max(ls[0], 2 ** round(math.log2(lmax + 1)) - 1))
    batch = max(1, min(_log_uniform(rng, *bs), most // (lmax + 1) ** 3))
    mres = rng.choice([1, 1, 1, 2, 3]) if lmax >= 63 else 1
    mmax = lmax // mres
    # the tightest grid, one a little larger, or one dealiased by 3/2, within what the family's path takes
    nlat = min(rng.choice([lmax + 1, lmax + 2 + lmax // 16, 3 * (lmax + 1) // 2]), max(lmax + 1, 1024))
    if rng.random() < 0.5:
        nphi = 2 ** math.ceil(math.log2(2 * mmax + 2))
    else:
        nphi = _smooth_nphi(rng.choice([2 * mmax + 2, 3 * mmax + 1]))
    return {"kind": kind, "dtype": dtype, "path": path, "lmax": lmax, "mmax": mmax, "nlat": nlat, "nphi": nphi,
            "batch": batch, "mres": mres}


def _sizes_of_uneven(case):
    """(lmax, nlat, nphi) of every field: truncations 63, 127, 255 and 511 drawn evenly."""
    ls = synthetic.uneven_truncations(case["batch"], (63, 127, 255, 511))
    return [(l, l + 1, 2 * (l + 1)) for l in ls]


def _degrees_orders(lmax, mmax, mres):
    n = np.concatenate([np.arange(k * mres, lmax + 1) for k in range(mmax + 1)])
    m = np.concatenate([np.full(lmax + 1 - k * mres, k * mres) for k in range(mmax + 1)])
    return n, m


def _spectra(gen, lmax, mmax, mres, batch, power, dtype):
    """Random spectra with a power law in n, real at m = 0."""
    n, m = (torch.from_numpy(v).cuda() for v in _degrees_orders(lmax, mmax, mres))
    a = torch.randn(2, batch, n.numel(), generator=gen, dtype=torch.float64, device="cuda")
    a *= (n.double() + 1.0) ** -power
    a[1, :, m == 0] = 0
    return torch.complex(a[0], a[1]).to(torch.complex128 if dtype == "f64" else torch.complex64)


def _grids(gen, nlat, nphi, batch, dtype):
    return torch.randn(batch, nlat, nphi, generator=gen, dtype=torch.float64, device="cuda").to(
        torch.float64 if dtype == "f64" else torch.float32)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    c, dt, b = case, case["dtype"], case["batch"]
    spec = lambda p: _spectra(gen, c["lmax"], c["mmax"], c["mres"], b, p, dt)      # noqa: E731
    grid = lambda: _grids(gen, c["nlat"], c["nphi"], b, dt)                       # noqa: E731
    if c["kind"] in ("scalar", "grad"):
        return {"spec": spec(1.0), "grid": grid()}
    if c["kind"] in ("vector", "vector_grad"):
        return {"S": spec(1.5), "T": spec(1.5), "vt": grid(), "vp": grid()}
    sizes = _sizes_of_uneven(c)
    return {"specs": [_spectra(gen, l, l, 1, 1, 1.0, dt)[0] for l, _, _ in sizes],
            "grids": [_grids(gen, la, ph, 1, dt)[0] for _, la, ph in sizes]}


def prepare(case, seed):
    state = _inputs(case, seed)
    state["kind"] = case["kind"]
    if case["kind"] == "uneven":
        sizes = _sizes_of_uneven(case)
        state["sht"] = UnevenBatch([s[0] for s in sizes], [s[1] for s in sizes], [s[2] for s in sizes],
                                   path=case["path"])
        # the fields' results side by side in one buffer per direction, kept from step to step
        for k in ("specs", "grids"):
            each = [v.numel() for v in state[k]]
            state[k + "_all"] = torch.empty(sum(each), dtype=state[k][0].dtype, device="cuda")
            state[k + "_out"] = [v.view(like.shape) for v, like in zip(state[k + "_all"].split(each), state[k])]
        return state
    path = {("f64", "cc"): {}, ("f32", "cc"): {}, ("f64", "tc"): {"fp64_path": "tc"},
            ("f32", "tc"): {"fp32_path": "tc"}}[case["dtype"], case["path"]]
    state["sht"] = SHT(case["lmax"], case["mmax"], case["nlat"], case["nphi"], mres=case["mres"], **path)
    for k in {"grad": ("spec",), "vector_grad": ("S", "T")}.get(case["kind"], ()):
        state[k].requires_grad_(True)
    return state


def run(state):
    sht, kind = state["sht"], state["kind"]
    if kind == "scalar":
        return sht.synth(state["spec"]), sht.analys(state["grid"])
    if kind == "vector":
        return sht.synth_vec(state["S"], state["T"]) + sht.analys_vec(state["vt"], state["vp"])
    if kind == "uneven":
        sht.synth_(state["specs"], out=state["grids_out"])
        sht.analys_(state["grids"], out=state["specs_out"])
        return state["grids_all"], state["specs_all"]
    if kind == "grad":
        loss = ((sht.synth(state["spec"]) - state["grid"]) ** 2).sum()
        return loss.detach(), torch.autograd.grad(loss, state["spec"])[0]
    vt, vp = sht.synth_vec(state["S"], state["T"])
    loss = ((vt - state["vt"]) ** 2).sum() + ((vp - state["vp"]) ** 2).sum()
    return (loss.detach(),) + torch.autograd.grad(loss, (state["S"], state["T"]))


def _work_of(lmax, mmax, mres, nlat, nphi, batch, elem, vector):
    """One transform in one direction: data in and out once; the Legendre sums
    (north/south folded: one real x complex multiply-add per degree, order,
    latitude pair and field, and the three-term recurrence once per degree, order
    and pair) and the real FFTs."""
    nlm = sum(lmax - k * mres + 1 for k in range(mmax + 1))
    pairs = (nlat + 1) // 2
    comps = 2 if vector else 1
    data = batch * comps * (2 * nlm + nlat * nphi) * elem
    sums = nlm * pairs * ((8 if vector else 4) + batch * (16 if vector else 4))
    fft = batch * comps * nlat * 2.5 * nphi * math.log2(max(nphi, 2))
    return data, sums + fft


def work(case):
    elem = 8 if case["dtype"] == "f64" else 4
    if case["kind"] == "uneven":
        each = [_work_of(l, l, 1, la, ph, 1, elem, False) for l, la, ph in _sizes_of_uneven(case)]
    else:
        each = [_work_of(case["lmax"], case["mmax"], case["mres"], case["nlat"], case["nphi"], case["batch"], elem,
                         case["kind"].startswith("vector"))]
    return {"bytes": 2 * sum(e[0] for e in each), "flops": 2 * sum(e[1] for e in each)}


# ---------------------------------------------------------------- 64-bit values


def _gauss(n):
    """Nodes (descending) and weights of the n-point Gauss-Legendre rule, by Newton's iteration."""
    i = np.arange(n)
    x = np.cos(np.pi * (i + 0.75) / (n + 0.5))
    for _ in range(8):
        p0, p1 = np.ones(n), x.copy()
        for k in range(2, n + 1):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
        d = n * (p0 - x * p1) / ((1 - x) * (1 + x))
        step = p1 / d
        x = x - step
        if np.abs(step).max() < 1e-15:
            break
    return x, 2 / ((1 - x) * (1 + x) * d * d)


class _Definition:
    """The transform by its definition in float64: orthonormal P_n^m at every
    latitude by the three-term recurrence (small values carried with a power of
    two apart), sums over the degrees or latitudes, and the longitude FFT."""

    SMALL = 2.0 ** -300

    def __init__(self, case):
        self.lmax, self.mmax, self.mres = case["lmax"], case["mmax"], case["mres"]
        self.nlat, self.nphi = case["nlat"], case["nphi"]
        x, w = _gauss(self.nlat)
        self.x, self.w = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
        self.st = torch.sqrt((1 - self.x) * (1 + self.x))
        # P_m^m = y 2^(-300 k) of every order
        y, k = np.full(self.nlat, math.sqrt(1 / (4 * math.pi))), np.zeros(self.nlat, dtype=np.int64)
        st = self.st.cpu().numpy()
        starts, ks = [], []
        for m in range(self.mmax * self.mres + 1):
            if m:
                y = y * st * math.sqrt((2 * m + 1) / (2 * m))
            small = y < self.SMALL
            y, k = np.where(small, y / self.SMALL, y), k + small
            if m % self.mres == 0:
                starts.append(y)
                ks.append(k)
        self.y0 = torch.from_numpy(np.array(starts)).cuda()
        self.k0 = torch.from_numpy(np.array(ks)).cuda()
        self.col = np.concatenate([[0], np.cumsum([self.lmax - j * self.mres + 1 for j in range(self.mmax + 1)])])
        self.nlm = int(self.col[-1])

    def blocks(self, vector=False):
        """Per block of orders: the order indices, the packed index [order, degree] of
        each coefficient (nlm where there is none), P and, for vectors, sin dP/dtheta
        [order, degree, latitude]."""
        first = 0
        while first <= self.mmax:
            deg = self.lmax - first * self.mres + 1
            count = max(1, min(self.mmax + 1 - first, (1 << 29) // (deg * self.nlat)))
            j = torch.arange(first, first + count, device="cuda")
            m = (j * self.mres).double()[:, None]
            y1, k = self.y0[j], self.k0[j]
            y2 = torch.zeros_like(y1)
            P = torch.zeros(count, deg, self.nlat, dtype=torch.float64, device="cuda")
            dP = torch.zeros_like(P) if vector else None
            for i in range(deg):
                n = m + i
                if i:
                    a = torch.sqrt((4 * n * n - 1) / (n * n - m * m))
                    b = torch.sqrt((2 * n + 1) / (2 * n - 3).clamp(min=1) * ((n - 1) ** 2 - m * m) / (n * n - m * m))
                    y1, y2 = a * self.x * y1 - b * y2, y1
                    big = (k > 0) & (y1.abs() >= 1)
                    y1, y2 = (torch.where(big, y * self.SMALL, y) for y in (y1, y2))
                    k = k - big.long()
                kept = k == 0
                P[:, i] = torch.where(kept, y1, 0.0)
                if not vector:
                    continue
                c = torch.sqrt((2 * n + 1) * (n * n - m * m) / (2 * n - 1).clamp(min=1)) if i else torch.zeros_like(m)
                dP[:, i] = torch.where(kept, n * self.x * y1 - c * y2, 0.0)
            i = torch.arange(deg, device="cuda")
            col = torch.from_numpy(self.col[first:first + count]).cuda()
            length = self.lmax - j * self.mres + 1
            index = torch.where(i[None] < length[:, None], col[:, None] + i[None], self.nlm)
            yield j, index, P, dP
            first += count

    @staticmethod
    def _sum(P, a):
        """sum over the middle axis of P [order, k, l] times complex a [batch, order, k]."""
        r = torch.view_as_real(a).permute(1, 2, 0, 3)
        out = torch.bmm(P.transpose(1, 2), r.reshape(r.shape[0], r.shape[1], -1))
        out = out.reshape(out.shape[0], out.shape[1], -1, 2).permute(2, 0, 1, 3)
        return torch.view_as_complex(out.contiguous())            # [batch, order, l]

    def _rows(self, F):
        """Real fields of the Fourier sums F [batch, order, latitude]."""
        full = torch.zeros(F.shape[0], self.nlat, self.nphi // 2 + 1, dtype=F.dtype, device="cuda")
        full[:, :, :self.mmax + 1] = F.transpose(1, 2)
        return torch.fft.irfft(full, n=self.nphi, dim=-1) * self.nphi

    def _orders(self, f):
        return torch.fft.rfft(f.double(), dim=-1)[..., :self.mmax + 1].transpose(1, 2)

    def _padded(self, a):
        """Spectra with a zero behind them for the indices that hold no coefficient."""
        a = a.detach().to(torch.complex128).clone()
        a[:, :self.lmax + 1].imag = 0
        return torch.cat([a, torch.zeros_like(a[:, :1])], dim=1)

    def _spec(self, batch):
        return torch.zeros(batch, self.nlm + 1, dtype=torch.complex128, device="cuda")

    def _finish(self, a):
        a[:, :self.lmax + 1].imag = 0
        return a[:, :self.nlm]

    def synth(self, a):
        a = self._padded(a)
        F = torch.zeros(a.shape[0], self.mmax + 1, self.nlat, dtype=torch.complex128, device="cuda")
        for j, index, P, _ in self.blocks():
            F[:, j] = self._sum(P, a[:, index])
        return self._rows(F)

    def _scaled_orders(self, f, weighted):
        """Weighted: the quadrature; else the transpose of the synthesis (orders m > 0 count twice)."""
        F = self._orders(f)
        if weighted:
            return F * (self.w * (2 * math.pi / self.nphi))
        twice = torch.full((self.mmax + 1, 1), 2.0, dtype=torch.float64, device="cuda")
        twice[0] = 1
        return F * twice

    def analys(self, f, weighted=True):
        F, out = self._scaled_orders(f, weighted), self._spec(f.shape[0])
        for j, index, P, _ in self.blocks():
            out[:, index.reshape(-1)] = self._sum(P.transpose(1, 2), F[:, j]).reshape(f.shape[0], -1)
        return self._finish(out)

    def synth_vec(self, S, T):
        S, T = self._padded(S), self._padded(T)
        vt = torch.zeros(S.shape[0], self.mmax + 1, self.nlat, dtype=torch.complex128, device="cuda")
        vp = torch.zeros_like(vt)
        for j, index, P, dP in self.blocks(vector=True):
            im = 1j * (j * self.mres).double()[:, None]
            s, t = S[:, index], T[:, index]
            vt[:, j] = (self._sum(dP, s) - im * self._sum(P, t)) / self.st
            vp[:, j] = (im * self._sum(P, s) + self._sum(dP, t)) / self.st
        return self._rows(vt), self._rows(vp)

    def analys_vec(self, ft, fp, weighted=True):
        vt, vp = (self._scaled_orders(f, weighted) / self.st for f in (ft, fp))
        S, T = self._spec(ft.shape[0]), self._spec(ft.shape[0])
        for j, index, P, dP in self.blocks(vector=True):
            im = 1j * (j * self.mres).double()[:, None]
            P, dP = P.transpose(1, 2), dP.transpose(1, 2)
            t, p = vt[:, j], vp[:, j]
            scale = torch.ones(1, dtype=torch.float64, device="cuda")
            if weighted:
                n = ((j * self.mres)[:, None] + torch.arange(index.shape[1], device="cuda")[None]).double()
                scale = (n > 0) / (n * (n + 1)).clamp(min=1)
            S[:, index.reshape(-1)] = (scale * (self._sum(dP, t) - im * self._sum(P, p))).reshape(ft.shape[0], -1)
            T[:, index.reshape(-1)] = (scale * (im * self._sum(P, t) + self._sum(dP, p))).reshape(ft.shape[0], -1)
        return self._finish(S), self._finish(T)


def exact(case, seed):
    inp = _inputs(case, seed)
    if case["kind"] == "uneven":
        sizes = _sizes_of_uneven(case)
        grids, specs = [None] * len(sizes), [None] * len(sizes)
        for size in sorted(set(sizes)):
            at = [i for i, s in enumerate(sizes) if s == size]
            d = _Definition(dict(case, lmax=size[0], mmax=size[0], nlat=size[1], nphi=size[2]))
            g = d.synth(torch.stack([inp["specs"][i] for i in at]))
            s = d.analys(torch.stack([inp["grids"][i] for i in at]))
            for q, i in enumerate(at):
                grids[i], specs[i] = g[q].reshape(-1), s[q]
        return torch.cat(grids), torch.cat(specs)
    d = _Definition(case)
    if case["kind"] == "scalar":
        return d.synth(inp["spec"]), d.analys(inp["grid"])
    if case["kind"] == "vector":
        return d.synth_vec(inp["S"], inp["T"]) + d.analys_vec(inp["vt"], inp["vp"])
    if case["kind"] == "grad":
        r = d.synth(inp["spec"]) - inp["grid"].double()
        return (r * r).sum(), d.analys(2 * r, weighted=False)
    vt, vp = d.synth_vec(inp["S"], inp["T"])
    rt, rp = vt - inp["vt"].double(), vp - inp["vp"].double()
    return ((rt * rt).sum() + (rp * rp).sum(),) + d.analys_vec(2 * rt, 2 * rp, weighted=False)
