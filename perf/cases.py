"""The work that a user of this library has it do, as cases that can be timed.

Each case is one record (or a set of channels) and one plan.  A pass is what the
library's user calls for every new record: ``ss_reset``, ``ss_accumulate`` over
the record, ``ss_finalize`` (or the allocation-free power spectrum), and the
spectra with their error bars kept as float32: the estimator's arithmetic up to
the sums over groups is float32 (the ABI's doubles carry float64 only across
groups), so a program that stores spectra keeps complex64 and float32.  Every
spectrum and every error bar is returned whole.

The plan is made once, in ``prepare``, as a program that processes many records
makes it; where such a program would let the library time its kernel forms first
(the long record), ``prepare`` does too.

``exact`` restates the estimator in float64 with plain torch operations: frames,
window, discrete Fourier transform with positive exponent, centring over the
group, the unbiased k-statistics, and the mean and standard error over groups.
"""
from __future__ import annotations

import math

import torch

import paper_2505_01231_gb300 as ps

# ---------------------------------------------------------------- the cases
# kind: "plan"    one plan, device-resident record (optionally several channels)
#       "stream"  the same from page-locked host memory in several chunks
#       "seq"     with the short-time spectra of blocks of groups as well
#       "complex" spectra of one complex-valued signal (two real channels)
#       "noalloc" power spectrum through the entry point that allocates nothing


def _case(name, kind, C, n, T, m, orders, precision, **kw):
    d = dict(name=name, kind=kind, channels=C, n=n, T=T, m=m, orders=orders, precision=precision,
             dtype="f32", window="hann", tune=False, chunks=1, block=0)
    d.update(kw)
    return d


def listed():
    return [
        # a short buffer's power spectrum inside a loop that must not allocate: launches and
        # latency are all there is
        _case("psd-noalloc-2^16-T256-m8", "noalloc", 1, 1 << 16, 256, 8, "2", "fp32"),
        # a short laboratory record with the plan's default precision, every order
        _case("short-2^20-T256-m10-fp32", "plan", 1, 1 << 20, 256, 10, "234", "fp32"),
        # the long record: 2^28 samples, 513 bins, full S2/S3/S4 grids in the split precision,
        # kernel forms timed by the plan first
        _case("long-2^28-T1024-m10-fp16x3", "plan", 1, 1 << 28, 1024, 10, "234", "fp16x3",
              tune=True),
        # a medium record of the same kind with the plan's default (float32) fourth order
        _case("mid-2^25-T1024-m10-fp32", "plan", 1, 1 << 25, 1024, 10, "234", "fp32"),
        # an odd length, longer frames in smaller groups, the confined Gaussian window
        _case("odd-5000003-T2048-m9-fp16x3", "plan", 1, 5000003, 2048, 9, "234", "fp16x3",
              window="acg"),
        # an ADC record streamed from page-locked host memory in odd-sized chunks
        _case("adc16-stream-2^26-T4096-m10-fp16x3", "stream", 1, 1 << 26, 4096, 10, "234",
              "fp16x3", dtype="i16", chunks=5),
        # a power spectrum alone of a long record: samples in, a few thousand numbers out
        _case("power-2^27-T2048-m16", "plan", 1, 1 << 27, 2048, 16, "2", "fp32"),
        # S2 and S3 only, short frames in large groups
        _case("bispec-8389385-T128-m32", "plan", 1, 8389385, 128, 32, "23", "fp32"),
        # four channels, every cross combination of every order, split precision
        _case("mc4-2^21-T512-m20-fp16x3", "plan", 4, 1 << 21, 512, 20, "234", "fp16x3"),
        # two channels, every cross combination, the plan's default precision
        _case("mc2-2^20-T256-m8-fp32", "plan", 2, 1 << 20, 256, 8, "234", "fp32"),
        # a non-stationary record: short-time spectra of every 64 groups beside the whole
        _case("seq-2^21-T128-m8-fp32", "seq", 1, 1 << 21, 128, 8, "234", "fp32", block=64),
        # one complex-valued signal: power, bispectrum and trispectrum cut on the whole plane
        _case("complex-2^19-T128-m8", "complex", 2, 1 << 19, 128, 8, "234", "fp32"),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["noalloc", "auto", "auto", "auto", "stream", "power", "bispec", "cross",
                       "cross", "seq", "complex"])
    win = rng.choice(["hann", "hann", "acg"])
    if kind == "noalloc":
        T = 2 ** rng.randint(6, 12)
        m = rng.randint(2, 16)
        return _nameless("noalloc", 1, logint(max(1 << 13, 3 * m * T), 1 << 21), T, m, "2", "fp32",
                         window=win)
    if kind == "auto":
        # the float32 fourth order takes any group size; the split one serves long frames
        prec = rng.choice(["fp32", "fp16x3"])
        T = 2 ** (rng.randint(6, 11) if prec == "fp32" else rng.randint(10, 12))
        m = rng.randint(5, 24) if prec == "fp32" else rng.randint(8, 10)
        top = (1 << 35 if prec == "fp32" else 1 << 37) // max(T, 256)
        return _nameless("plan", 1, logint(max(1 << 16, 4 * m * T), top), T, m, "234", prec,
                         window=win, dtype=rng.choice(["f32", "f32", "i16"]))
    if kind == "stream":
        T, m = 2 ** rng.randint(10, 12), rng.randint(8, 10)
        return _nameless("stream", 1, logint(1 << 21, (1 << 37) // T), T, m, "234", "fp16x3",
                         dtype=rng.choice(["i16", "f32"]), chunks=rng.randint(2, 7))
    if kind == "power":
        T, m = 2 ** rng.randint(5, 12), rng.randint(2, 32)
        return _nameless("plan", 1, logint(1 << 20, 1 << 27), T, m, "2", "fp32", window=win,
                         dtype=rng.choice(["f32", "i16"]))
    if kind == "bispec":
        T, m = 2 ** rng.randint(5, 9), rng.randint(4, 48)
        return _nameless("plan", 1, logint(1 << 18, 1 << 24), T, m, "23", "fp32", window=win)
    if kind == "cross":
        C, T, prec = rng.randint(2, 4), 2 ** rng.randint(6, 9), rng.choice(["fp32", "fp16x3", "tf32x3"])
        m = rng.randint(5, 24)
        top = (1 << 21 if prec != "fp32" and C == 4 else 1 << 19 if C > 2 else 1 << 20)
        return _nameless("plan", C, logint(max(1 << 15, 4 * m * T), top), T, m, "234", prec)
    if kind == "seq":
        T, m = 2 ** rng.randint(5, 8), rng.randint(5, 16)
        return _nameless("seq", 1, logint(1 << 18, 1 << 22), T, m, "234", "fp32",
                         block=rng.randint(24, 160))
    T, m = 2 ** rng.randint(5, 7), rng.randint(5, 16)
    return _nameless("complex", 2, logint(1 << 15, 1 << 19), T, m, "234", "fp32")


def _nameless(*a, **kw):
    d = _case("", *a, **kw)
    del d["name"]
    return d


# ---------------------------------------------------------------- inputs
def _lowpass(y, phi, span):
    """y_t <- sum_{k < span} phi^k y_{t-k} (span a power of two), along the last axis."""
    s = 1
    while s < span:
        z = y.clone()
        z[..., s:].add_(y[..., :-s], alpha=phi ** s)
        y, s = z, 2 * s
    return y


def _record(case, seed):
    """[channels][n] samples on the GPU: a low-passed Gaussian with a quadratic part (so that S3
    and S4 are there to be found), several channels with a shared part, or 16-bit ADC samples
    of a low-passed telegraph signal with noise."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    C, n = case["channels"], case["n"]

    def normal():
        return torch.randn(n, generator=g, device="cuda")

    if case["dtype"] == "i16":
        flips = torch.rand(n, generator=g, device="cuda") < 1e-3
        s = 1.0 - 2.0 * (torch.cumsum(flips, 0, dtype=torch.int32) & 1).float()
        s = _lowpass(s, 0.73, 32) * 0.27
        return torch.clamp(torch.round(2000.0 * s + 800.0 * normal()), -32768, 32767).to(torch.int16)[None]
    if C == 1:
        y = _lowpass(normal(), 0.9, 128)
        return (y + 0.3 * (y * y - 1.0))[None]
    shared = _lowpass(normal(), 0.95, 128)
    return torch.stack([shared + 0.5 * normal() + 0.2 * (1 + 0.2 * c) * shared * shared
                        for c in range(C)])


# the complex case: one signal z = x + j y of channels 0 and 1; its power, S3 and S4 cut
_Z, _ZC = (0, 1, 0), (0, 1, 1)
_RECORDS = [(2, _Z, _ZC), (3, _Z, _Z, _ZC), (4, _Z, _ZC, _Z, _ZC)]
_SIGMA = 0.14


def prepare(case, seed):
    st = dict(case)
    x = _record(case, seed)
    if case["kind"] == "stream":
        host = torch.empty(x.shape, dtype=x.dtype, pin_memory=True)
        host.copy_(x)
        torch.cuda.synchronize()
        x = host
    st["x"] = x
    M = case["T"] // 2 + 1
    if case["kind"] == "noalloc":
        st["keys"] = [("S2", (M, 2)), ("S2_err", (M, 2))]
        st["out"] = torch.empty(4 * M, dtype=torch.float64, device="cuda")
        return st
    orders = tuple(int(o) for o in case["orders"])
    if case["kind"] == "complex":
        plan = ps.Plan(channels=case["channels"], T=case["T"], dt=0.5, m=case["m"], orders=(2,),
                       combos=[(2, 0, 0, -1, -1)])
        ps.ss_set_complex(plan.handle, _RECORDS, 0)
        size = ps.ss_complex_size(plan.handle)
        st["out"] = torch.empty(2 * size, dtype=torch.float64, device="cuda")
    else:
        plan = ps.Plan(channels=case["channels"], T=case["T"], dt=0.5, m=case["m"],
                       window=case["window"], sigma_t=_SIGMA, orders=orders, dtype=case["dtype"],
                       precision=case["precision"])
        if case["tune"]:
            ps.ss_autotune(plan.handle)
        # one device buffer for all spectra and error bars, in the order S2, S2_err, S3, ...
        shapes, keys = plan.shapes(), []
        for o in orders:
            keys += [("S%d" % o, shapes["S%d" % o]), ("S%d_err" % o, shapes["S%d" % o])]
        st["keys"] = [(k, tuple(s) + (2,)) for k, s in keys]
        st["out"] = torch.empty(sum(math.prod(s) for _, s in st["keys"]), dtype=torch.float64,
                                device="cuda")
        if case["kind"] == "seq":
            blocks = case["n"] // (case["T"] * case["m"]) // case["block"]
            per_block, _ = ps.ss_sequential_info(plan.handle)
            st["blocks"] = torch.empty(per_block * blocks, dtype=torch.float64, device="cuda")
            ps.ss_set_sequential(plan.handle, case["block"], st["blocks"], blocks)
    st["plan"] = plan
    return st


def _views(flat, keys):
    out, o = {}, 0
    for k, shape in keys:
        c = math.prod(shape)
        out[k] = flat[o:o + c].view(shape)
        o += c
    return out


def run(st):
    if st["kind"] == "noalloc":
        d = _views(st["out"], st["keys"])
        ps.ss_s2_noalloc(st["x"], st["n"], st["T"], 0.5, st["m"],
                         ps.SS_WIN_ACG if st["window"] == "acg" else ps.SS_WIN_HANN, _SIGMA,
                         d["S2"], d["S2_err"])
        return _views(st["out"].float(), st["keys"])
    plan, x = st["plan"], st["x"]
    plan.reset()
    if st["kind"] == "stream":
        # chunks of unequal, odd sizes: the plan carries the samples between groups over
        n, c = st["n"], st["chunks"]
        cuts = [0] + [(n * i) // c + 37 * i - 1 for i in range(1, c)] + [n]
        for a, b in zip(cuts, cuts[1:]):
            plan.accumulate(x[0, a:b])
    else:
        plan.accumulate(x)
    if st["kind"] == "complex":
        size = st["out"].numel() // 2
        ps.ss_finalize_complex(plan.handle, st["out"][:size], st["out"][size:])
        flat = st["out"].float()
        n1 = st["T"] + 1  # 2 M - 1 bins from -(M - 1) to M - 1
        shapes = [(n1, 2), (n1, n1, 2), (n1, n1, 2)]
        return _views(flat, [("S%d%s" % (o + 2, e), s) for e in ("", "_err")
                             for o, s in enumerate(shapes)])
    d = _views(st["out"], st["keys"])
    ps.ss_finalize(plan.handle, d.get("S2"), d.get("S3"), d.get("S4"), d.get("S2_err"),
                   d.get("S3_err"), d.get("S4_err"))
    out = _views(st["out"].float(), st["keys"])
    if st["kind"] == "seq":
        out["blocks"] = st["blocks"].float()
    return out


# ---------------------------------------------------------------- work
def _combos(C):
    pairs = [(a, b) for a in range(C) for b in range(a, C)]
    return {2: pairs,
            3: [(a, b, c) for a in range(C) for b in range(a, C) for c in range(b, C)],
            4: [pairs[i] + pairs[j] for i in range(len(pairs)) for j in range(i, len(pairs))]}


def work(case):
    """Every sample read once, every spectrum and error bar (double, as the ABI writes it) written
    once; the transform (2.5 T log2 T a frame), 14 operations a frame and grid point of S3 and 10 of
    the one-channel S4 (40 with several channels, 44 for complex operands), over the points that the
    symmetries leave."""
    C, T, m, n = case["channels"], case["T"], case["m"], case["n"]
    M, frames = T // 2 + 1, (n // (T * m)) * m
    nbytes = n * C * (2 if case["dtype"] == "i16" else 4)
    flops = C * frames * 2.5 * T * math.log2(T)
    cb = _combos(C)
    if case["kind"] == "complex":
        p1 = 2 * M - 1
        nbytes += 32 * (p1 + 2 * p1 * p1)
        flops += frames * (8 * p1 + 14 * (p1 * p1 - M * (M - 1)) + 44 * p1 * p1)
        return {"bytes": float(nbytes), "flops": float(flops)}
    outs = 0
    for o in (int(c) for c in case["orders"]):
        k = len(cb[o])
        if o == 2:
            outs += k * M
            flops += k * frames * M * (4 if C == 1 else 8)
        elif C == 1:
            outs += M * M
            h = (M - 1) // 2
            pts = sum(M - 2 * i for i in range(h + 1)) if o == 3 else M * (M + 1) // 2
            flops += frames * pts * (14 if o == 3 else 10)
        else:
            outs += k * (2 * M - 1) * M
            pts = (2 * M - 1) * M - (M * (M - 1) // 2 if o == 3 else 0)
            flops += k * frames * pts * (14 if o == 3 else 40)
    blocks = n // (T * m) // case["block"] if case["block"] else 0
    return {"bytes": float(nbytes + 32 * outs * (1 + blocks)), "flops": float(flops)}


# ---------------------------------------------------------------- float64
def _window(case):
    T = case["T"]
    i = torch.arange(T, dtype=torch.float64, device="cuda")
    if case["window"] == "hann":
        return 0.5 - 0.5 * torch.cos(2 * math.pi * i / T)
    mid, d = (T - 1) / 2, 4.0 * T * T * _SIGMA * _SIGMA

    def G(x):
        return torch.exp(-(x - mid) ** 2 / d)

    h = torch.tensor(-0.5, dtype=torch.float64, device="cuda")
    return G(i) - G(h) * (G(i + T) + G(i - T)) / (G(h + T) + G(h - T))


def _centred(x, case, g, a, b):
    """Centred coefficients [C, b - a groups, m, M] of groups a..b."""
    T, m = case["T"], case["m"]
    z = x[:, a * m * T:b * m * T].double().view(x.shape[0], b - a, m, T) * g
    d = torch.fft.rfft(z, dim=-1).conj()  # positive exponent
    return (d - d.mean(2, keepdim=True)).resolve_conj().contiguous()


class _Sums:
    """Sums over groups of Re, Im and their squares, at one set of points."""

    def __init__(self, shape):
        self.s = torch.zeros((4,) + tuple(shape), dtype=torch.float64, device="cuda")

    def add(self, idx, v):
        """v [groups, ...] complex or real, added at index idx."""
        re = v.real if v.is_complex() else v
        self.s[(0,) + idx] += re.sum(0)
        self.s[(2,) + idx] += (re * re).sum(0)
        if v.is_complex():
            self.s[(1,) + idx] += v.imag.sum(0)
            self.s[(3,) + idx] += (v.imag * v.imag).sum(0)

    def done(self, G, norm):
        mean = self.s[:2] / G
        var = torch.clamp(self.s[2:] / G - mean * mean, min=0) / (G - 1)
        return (torch.movedim(mean * norm, 0, -1).contiguous(),
                torch.movedim(var.sqrt() * norm, 0, -1).contiguous())


def _c4(x, y, z, w, m):
    """c4 at (row, column) pairs: x, y [G, m, R], z, w [G, m, L] centred."""
    def dot(p, q):
        return torch.bmm(p.transpose(1, 2), q)

    xy, zw = x * y, z * w
    t = (xy.sum(1)[:, :, None] * zw.sum(1)[:, None, :]).add_(dot(x, z).mul_(dot(y, w)))
    t.add_(dot(x, w).mul_(dot(y, z)))
    return dot(xy, zw).mul_(m * (m + 1)).sub_(t.mul_(m - 1)).div_((m - 1) * (m - 2) * (m - 3))


def _add_one_channel(d, m, orders, sums):
    M = d.shape[-1]
    p = d.real ** 2 + d.imag ** 2
    sums["S2"].add((0,), p.sum(1) / (m - 1))
    if "3" in orders:
        pref = m / ((m - 1) * (m - 2))
        for k in range((M - 1) // 2 + 1):  # k <= l, k + l <= M - 1
            v = (d[:, :, k:k + 1] * d[:, :, k:M - k] * d[:, :, 2 * k:].conj()).sum(1) * pref
            sums["S3"].add((0, k, slice(k, M - k)), v)
    if "4" in orders:
        step = max(1, int(6e8 / (32 * M * M)))
        for a in range(0, d.shape[0], step):
            e, q = d[a:a + step], p[a:a + step]
            r = torch.cat([e.real, e.imag], -1)
            r = torch.bmm(r.transpose(1, 2), r).square_()  # [*, 2M, 2M] real products
            uv = (r[:, :M, :M] + r[:, M:, M:]).add_(r[:, :M, M:]).add_(r[:, M:, :M]).mul_(2)
            s = q.sum(1)
            uv.add_(s[:, :, None] * s[:, None, :])
            c4 = torch.bmm(q.transpose(1, 2), q).mul_(m * (m + 1)).sub_(uv.mul_(m - 1))
            sums["S4"].add((0,), c4.div_((m - 1) * (m - 2) * (m - 3)))


def _full(d):
    """Half spectrum [.., M] to bins -(M-1)..M-1 of a real signal."""
    return torch.cat([d[..., 1:].flip(-1).conj(), d], -1)


def _add_channels(d, m, orders, sums):
    C, M = d.shape[0], d.shape[-1]
    f, cb = [_full(d[c]) for c in range(C)], _combos(C)
    for i, (a, b) in enumerate(cb[2]):
        sums["S2"].add((i,), (d[a] * d[b].conj()).sum(1) / (m - 1))
    n1 = 2 * M - 1
    for i, (a, b, c) in enumerate(cb[3]):
        for l in range(M):
            v = (f[a][:, :, :n1 - l] * d[b][:, :, l:l + 1] * f[c][:, :, l:].conj()).sum(1)
            sums["S3"].add((i, slice(0, n1 - l), l), v * (m / ((m - 1) * (m - 2))))
    step = max(1, int(1e9 / (16 * n1 * M)))
    for i, (a, b, c, e) in enumerate(cb[4]):
        for g in range(0, d.shape[1], step):
            s = slice(g, g + step)
            sums["S4"].add((i,), _c4(f[a][s], f[b][s].conj(), d[c][s], d[e][s].conj(), m))


def _add_complex(d, m, sums):
    fx, fy = _full(d[0]), _full(d[1])
    z, zc = fx + 1j * fy, fx - 1j * fy  # z and the transform of z* at each signed bin
    n1 = z.shape[-1]
    M = (n1 + 1) // 2
    rev = zc.flip(-1)  # z* at -k
    sums["S2"].add((), (z * rev).sum(1) / (m - 1))
    for r in range(n1):  # k = r - (M-1): columns with |k + l| <= M - 1
        lo, hi = max(0, M - 1 - r), min(n1, n1 + M - 1 - r)
        t = slice(r + lo - (M - 1), r + hi - (M - 1))
        v = (z[:, :, r:r + 1] * z[:, :, lo:hi] * rev[:, :, t]).sum(1)
        sums["S3"].add((r, slice(lo, hi)), v * (m / ((m - 1) * (m - 2))))
    step = max(1, int(1e9 / (16 * n1 * n1)))
    for g in range(0, z.shape[0], step):
        s = slice(g, g + step)
        sums["S4"].add((), _c4(z[s], rev[s], z[s], rev[s], m))


def exact(case, seed):
    x = _record(case, seed)
    C, T, m = case["channels"], case["T"], case["m"]
    M, G = T // 2 + 1, case["n"] // (T * m)
    g, dt, kind = _window(case), 0.5, case["kind"]
    # dt c2(X) / sum g^2 and so on: the Fourier coefficients are dt X
    norm = {"S2": dt / (g ** 2).sum(), "S3": dt ** 2 / (g ** 3).sum(), "S4": dt ** 3 / (g ** 4).sum()}
    cb, n1 = _combos(C), 2 * M - 1
    keys = ["S%s" % o for o in case["orders"]]
    if kind == "complex":
        shapes = {"S2": (n1,), "S3": (n1, n1), "S4": (n1, n1)}
    elif kind == "noalloc":
        shapes = {"S2": (1, M)}
    else:
        rows = M if C == 1 else n1
        shapes = {"S2": (len(cb[2]), M), "S3": (len(cb[3]), rows, M), "S4": (len(cb[4]), rows, M)}

    def estimate(ga, gb):
        sums = {k: _Sums(shapes[k]) for k in keys}
        step = max(1, int(2e9 / (16 * C * m * T)))
        for a in range(ga, gb, step):
            d = _centred(x, case, g, a, min(gb, a + step))
            if kind == "complex":
                _add_complex(d, m, sums)
            elif C == 1:
                _add_one_channel(d[0], m, case["orders"], sums)
            else:
                _add_channels(d, m, case["orders"], sums)
        res = {}
        for k in keys:
            mean, err = sums[k].done(gb - ga, norm[k])
            if k == "S3" and C == 1:  # computed on k <= l
                for v in (mean, err):
                    low = v.transpose(1, 2).clone()
                    eye = torch.arange(M, device="cuda")
                    low[:, eye, eye] = 0
                    v += low
            res[k], res[k + "_err"] = mean, err
        return res

    res = estimate(0, G)
    if kind == "noalloc":
        return {k: v[0] for k, v in res.items()}
    if kind == "complex":
        return {k + e: res[k + e] for e in ("", "_err") for k in keys}
    if kind == "seq":
        B, parts = case["block"], []
        for b in range(G // B):
            r = estimate(b * B, (b + 1) * B)
            parts += [r[k + e].reshape(-1) for k in keys for e in ("", "_err")]
        res["blocks"] = torch.cat(parts)
    return res
