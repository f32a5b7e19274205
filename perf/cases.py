"""Cases of the alignment library's performance: what a user has it do.

Every case goes through the public Python entry points
(``swalign.Aligner``, ``swalign.Bank``, ``uneven.UnevenGraph``).  ``kind``
names the entry point:

  pair     align_all_rotations: one pair, the whole curve over the rotations
  batch    align_batch: every query against every template
  bank     Bank.align: a request's queries against a device-resident bank
  uneven   UnevenGraph.replay: a batch of several image sizes as one graph
  stages   project, then quantiles: the rows and quantile functions themselves

The images are mixtures of anisotropic Gaussian blobs and rotated, shifted,
smoothly warped, noisy copies of them, clipped and normalised to unit mass
(``data = "blobs"``), or uniform random dense images (``"dense"``).

A sw_result is returned as two views of its bytes: the four 4-byte words
best_l, status, angle_rad (as bits) and template_index, and the three
doubles shift[0], shift[1] and d2.
"""
from __future__ import annotations

import math

import torch

from paper_2503_13756_gb300 import swalign, uneven

DEV = "cuda:0"
UNEVEN_SIZES = (64, 96, 128, 192, 256)
UNEVEN_WEIGHTS = (0.3, 0.25, 0.2, 0.15, 0.1)


def _case(kind, L, n, M, Nq, Nt, name=None, **kw):
    c = {"kind": kind, "L": L, "n": n, "M": M, "Nq": Nq, "Nt": Nt, "precision": "fp32",
         "metric": "sw2", "projector": "slice", "translation": 1, "level_rule": 0,
         "shift_grid": 0, "mode": 0, "q_L": L, "data": "blobs"}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call of the paper's timing setting: one pair of random
        # dense images, rotation only, L = n = M, the default projector
        _case("pair", 32, 32, 32, 1, 1, "dense_pair_32", data="dense", translation=0,
              projector="splat"),
        # an interactive alignment: one 64 x 64 pair, every rotation at 1
        # degree and the optimal translation
        _case("pair", 64, 360, 128, 1, 1, "single_pair_64"),
        # a small many-to-many batch at reduced precision
        _case("batch", 128, 256, 128, 64, 16, "batch_bf16_64x16", precision="bf16"),
        # ragged sizes on the direct projector, best template per query, the
        # translation restricted to a half-pixel grid
        _case("batch", 101, 240, 101, 301, 37, "ragged_splat_301x37", projector="splat", mode=1,
              shift_grid=32),
        # the ramp-filtered distance over a batch
        _case("batch", 128, 256, 128, 512, 64, "rfsw2_512x64", metric="rfsw2"),
        # the max-sliced distance over a small batch
        _case("batch", 128, 256, 128, 128, 16, "msw2_128x16", metric="msw2"),
        # particle images against one reference
        _case("batch", 128, 512, 256, 10000, 1, "one_reference_10000"),
        # the benchmark: many queries against many templates
        _case("batch", 128, 256, 128, 4096, 256, "many_to_many_4096x256"),
        # a batch of mixed image sizes, 64 templates of each, M = L, as one graph
        _case("uneven", 256, 256, 256, 2000, 64, "uneven_2000", precision="bf16"),
        # a served request of a few half-size images against the bank
        _case("bank", 256, 360, 256, 3, 1000, "serve_3_half_size", precision="bf16", q_L=128,
              mode=1),
        # a served batch at its largest, full-size images
        _case("bank", 256, 360, 256, 128, 1000, "serve_128_full_size", mode=1),
        # rows and quantile functions of a set of images, for a store
        _case("stages", 192, 256, 192, 64, 1, "rows_quantiles_192"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("pair", "batch", "batch", "batch", "bank", "uneven", "stages"))
    projector = rng.choice(("slice", "slice", "splat"))
    n = rng.choice((60, 64, 96, 120, 128, 180, 200, 240, 256, 320, 360, 384, 480, 512))
    if kind == "uneven":
        return _case(kind, 256, rng.choice((128, 256, 360)), 256, _log_int(rng, 200, 4000),
                     _log_int(rng, 4, 64), precision=rng.choice(("bf16", "fp16", "fp32")),
                     mode=rng.choice((0, 1)))
    L = _log_int(rng, 24, 256)
    M = min(256, max(16, _log_int(rng, 0.6 * L, 1.7 * L)))
    kw = {"projector": projector, "translation": rng.choice((1, 1, 1, 0)),
          "level_rule": rng.choice((0, 0, 0, 1)),
          "data": rng.choice(("blobs", "blobs", "blobs", "dense"))}
    if kind == "pair":
        return _case(kind, L, n, M, 1, 1, metric=rng.choice(("sw2", "sw2", "rfsw2")), **kw)
    if kind == "stages":
        return _case(kind, L, n, M, _log_int(rng, 1, 1024), 1,
                     metric=rng.choice(("sw2", "sw2", "rfsw2")), **kw)
    kw["precision"] = rng.choice(("fp32", "fp32", "bf16", "fp16", "fp32_simt"))
    kw["mode"] = rng.choice((0, 1))
    if kind == "bank":
        L += L & 1
        half = rng.choice((0, 1))
        return _case(kind, L, n, M, _log_int(rng, 1, 128), _log_int(rng, 16, 1000),
                     q_L=L // 2 if half else L, **kw)
    metric = rng.choice(("sw2", "sw2", "sw2", "rfsw2", "msw2"))
    if metric == "msw2":  # O(n^2 M) per pair
        n = min(n, 256)
        return _case(kind, L, n, min(M, 128), _log_int(rng, 2, 128), _log_int(rng, 1, 16),
                     metric=metric, **kw)
    kw["shift_grid"] = rng.choice((0, 0, 32)) if kw["translation"] else 0
    c = _case(kind, L, n, M, _log_int(rng, 4, 4096), _log_int(rng, 1, 256), metric=metric, **kw)
    while work(c)["flops"] > 4e10:  # at most about the benchmark's time
        c["Nq"] -= c["Nq"] // 4
    return c


# --------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _mixtures(g, count, L):
    """Blob mixtures: centres in the central 40/64 of the image, widths 3-8 px
    and weights of 2 to 6 blobs at L = 64, scaled with L."""
    s = L / 64.0

    def u(*shape):
        return torch.rand(shape, generator=g, device=DEV)

    k = torch.randint(2, 7, (count, 1), generator=g, device=DEV)
    w = (0.5 + 0.5 * u(count, 6)) * (torch.arange(6, device=DEV)[None] < k)
    return {"mu": (u(count, 6, 2) - 0.5) * 40.0 * s, "sd": (3.0 + 5.0 * u(count, 6, 2)) * s,
            "phi": math.pi * u(count, 6), "w": w}


def _render(g, mix, L, copies, noise=0.0):
    """Images of the mixtures; copies: turned by a random angle, shifted by
    whole pixels, warped by a smooth field, with noise."""
    count = mix["w"].shape[0]
    out = torch.empty((count, L, L), device=DEV)
    x = torch.arange(L, device=DEV, dtype=torch.float32) + 0.5 - L / 2
    step = max(1, (1 << 25) // (L * L))
    for c0 in range(0, count, step):
        sl = slice(c0, min(count, c0 + step))
        m = sl.stop - c0

        def u(*shape):
            return torch.rand(shape, generator=g, device=DEV)

        X = x[None, None, :].expand(m, L, L)
        Y = x[None, :, None].expand(m, L, L)
        if copies:
            amp = 3.0 * L / 128.0
            f = (0.5 + 1.5 * u(m, 4, 1, 1)) * 2.0 * math.pi / L
            p = 2.0 * math.pi * u(m, 4, 1, 1)
            t = torch.round((u(m, 2, 1, 1) - 0.5) * 16.0 * L / 128.0)
            b = 2.0 * math.pi * u(m, 1, 1)
            xs = X - t[:, 0] + amp * torch.sin(f[:, 0] * X + p[:, 0]) * torch.sin(f[:, 1] * Y + p[:, 1])
            ys = Y - t[:, 1] + amp * torch.sin(f[:, 2] * X + p[:, 2]) * torch.sin(f[:, 3] * Y + p[:, 3])
            X, Y = torch.cos(b) * xs + torch.sin(b) * ys, torch.cos(b) * ys - torch.sin(b) * xs
        acc = torch.zeros((m, L, L), device=DEV)
        for q in range(6):
            c = torch.cos(mix["phi"][sl, q])[:, None, None]
            s = torch.sin(mix["phi"][sl, q])[:, None, None]
            dx = X - mix["mu"][sl, q, 0][:, None, None]
            dy = Y - mix["mu"][sl, q, 1][:, None, None]
            e0 = (c * dx + s * dy) / mix["sd"][sl, q, 0][:, None, None]
            e1 = (c * dy - s * dx) / mix["sd"][sl, q, 1][:, None, None]
            acc += mix["w"][sl, q][:, None, None] * torch.exp(-0.5 * (e0 * e0 + e1 * e1))
        if copies and noise:
            acc += noise * torch.randn((m, L, L), generator=g, device=DEV)
        acc.clamp_(min=0.0)
        out[sl] = acc / acc.sum((1, 2), keepdim=True)
    return out


def _images(g, Nq, Nt, L, data, noise, q_L=None):
    """Queries and templates (queries at side q_L)."""
    q_L = L if q_L is None else q_L
    if data == "dense":
        return (torch.rand((Nq, q_L, q_L), generator=g, device=DEV),
                torch.rand((Nt, L, L), generator=g, device=DEV))
    mix = _mixtures(g, Nt, L)
    t = _render(g, mix, L, False)
    src = torch.randint(0, Nt, (Nq,), generator=g, device=DEV)
    qm = {k: v[src] for k, v in mix.items()}
    if q_L != L:
        qm["mu"], qm["sd"] = qm["mu"] * (q_L / L), qm["sd"] * (q_L / L)
    return _render(g, qm, q_L, True, noise), t


def _inputs(case, seed):
    """Device images of a case: (queries, templates), or one pair of them per
    size of an uneven batch."""
    g = _generator(seed)
    noise = 0.01 if case["kind"] in ("pair", "bank") else (0.02 if case["Nt"] == 1 else 0.0)
    if case["kind"] != "uneven":
        return _images(g, case["Nq"], case["Nt"], case["L"], case["data"], noise, case["q_L"])
    out = {}
    for L, w in zip(UNEVEN_SIZES, UNEVEN_WEIGHTS):
        out[L] = _images(g, max(1, round(case["Nq"] * w)), case["Nt"], L, case["data"], noise)
    return out


def _params(case, L=None, M=None):
    return swalign.make_params(
        L or case["L"], case["n"], M or case["M"], translation=case["translation"],
        level_rule=case["level_rule"], precision=case["precision"], metric=case["metric"],
        projector=case["projector"], shift_grid=case["shift_grid"],
        shift_step_q=8 if case["shift_grid"] else 0)


def _fields(out):
    """(words, doubles) of a buffer of sw_result, as views."""
    return out.view(torch.int32)[:, :4], out.view(torch.float64)[:, 2:]


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "mode": case["mode"]}
    if kind == "uneven":
        ins = _inputs(case, seed)
        b = [uneven.Bucket(L, _params(case, L, L), q, t) for L, (q, t) in ins.items()]
        s["graph"] = uneven.UnevenGraph(b, mode=case["mode"])
        s["fields"] = {str(k.L): _fields(k.out) for k in s["graph"].buckets}
        return s
    p = s["params"] = _params(case)
    s["q"], s["t"] = _inputs(case, seed)
    al = s["al"] = swalign.Aligner()
    Nq, Nt = case["Nq"], case["Nt"]
    if kind in ("batch", "pair"):
        al.reserve(p, Nq, Nt)
    elif kind == "bank":
        s["bank"] = swalign.Bank(al, s["t"], p)
        al.reserve(p, Nq, Nt)
        s["q_L"] = case["q_L"]
    if kind in ("batch", "bank"):
        rows = Nq * Nt if case["mode"] == 0 else Nq
        s["out"] = torch.empty((rows, 40), dtype=torch.uint8, device=DEV)
        s["fields"] = _fields(s["out"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "pair":
        D, S, best = s["al"].align_all_rotations(s["q"][0], s["t"][0], s["params"])
        return {"curve": D, "shifts": S, "best": _fields(best.view(1, 40))}
    if kind == "batch":
        s["al"].align_batch(s["q"], s["t"], s["params"], mode=s["mode"], out=s["out"])
        return s["fields"]
    if kind == "bank":
        s["bank"].align(s["q"], q_L=s["q_L"], mode=s["mode"], out=s["out"])
        return s["fields"]
    if kind == "uneven":
        s["graph"].replay()
        return s["fields"]
    rows, scale = s["al"].project(s["q"], s["params"], scale=True)
    q, center, norm = s["al"].quantiles(rows, s["params"])
    return {"rows": rows, "scale": scale, "quantiles": q, "center": center, "norm": norm}


# ----------------------------------------------------------------------- work
def _sizes(case):
    """(L, q_L, M, Nq, Nt) of every size of the case."""
    if case["kind"] == "uneven":
        return [(L, L, L, max(1, round(case["Nq"] * w)), case["Nt"])
                for L, w in zip(UNEVEN_SIZES, UNEVEN_WEIGHTS)]
    return [(case["L"], case["q_L"], case["M"], case["Nq"], case["Nt"])]


def work(case):
    """Bytes: the images (for a bank, its spectra at the precision's width)
    read once and the outputs written once.  Flops: FFTs at 5 N log2 N, the
    slice projection's grid FFTs and 9 x 9 taps (4 flops each) per slice
    sample or the splat's 8 per cell and angle, the correlation at 8 per
    (level, frequency, pair) and one real inverse FFT per pair (max-sliced:
    3 n^2 M per pair)."""
    n, nb, fl = case["n"], 0.0, 0.0
    kind, parts = case["kind"], 2 if case["metric"] == "rfsw2" else 1
    for L, q_L, M, Nq, Nt in _sizes(case):
        B = swalign.bins_of(_params(case, L, M))
        if case["projector"] == "slice":
            fft = 5.0 * B * math.log2(B)
            per = fft * (L / 2 + B / 2 + 9 + n / 4) + 4.0 * 81 * (n / 2) * (B / 2 + 1)
        else:
            per = 8.0 * L * L * n / 2
        if parts == 2:
            per += (n / 2) * 5.0 * B * math.log2(B)
        per += (n / 2) * B + 4.0 * (n / 2) * M * parts  # prefix sums, interpolation
        if kind == "stages":
            nb += Nq * (4.0 * q_L * q_L + 8 + 4.0 * n * B + parts * (4.0 * n * M + 24))
            fl += Nq * (per + parts * 5.0 * n * M)
            continue
        spec = parts * M / 2 * 5.0 * n * math.log2(n)
        images = Nq + (0 if kind == "bank" else Nt)
        pairs = float(Nq) * Nt
        nb += 4.0 * Nq * q_L * q_L
        if kind == "bank":
            width = 2 if case["precision"] in ("bf16", "fp16") else 4
            nb += Nt * (n / 2) * 2 * M * parts * width
        else:
            nb += 4.0 * Nt * L * L
        nb += 40.0 * (pairs if case["mode"] == 0 else Nq) + (24.0 * n if kind == "pair" else 0)
        if case["metric"] == "msw2":
            fl += images * per + pairs * 3.0 * n * n * M
        else:
            fl += images * (per + spec) + pairs * (8.0 * M * parts * (n / 2) +
                                                   2.5 * n * math.log2(n))
    return {"bytes": nb, "flops": fl}


# ---------------------------------------------------------------------- exact
def _rows64(img, L, n, B, case):
    """Projection rows [N][n][B] of FP64 images."""
    N, nh, h = img.shape[0], n // 2, 2.0 / L
    th = 2.0 * math.pi * torch.arange(nh, device=DEV, dtype=torch.float64) / n
    co, si = torch.cos(th), torch.sin(th)
    x = torch.arange(L, device=DEV, dtype=torch.float64) + 0.5 - L / 2  # in cells
    img = img.clamp(min=0.0)
    out = torch.zeros((N, nh, B), device=DEV, dtype=torch.float64)
    if case["projector"] == "splat":
        flat = img.reshape(N, L * L)
        for k in range(nh):
            u = (co[k] * x[None, :] + si[k] * x[:, None]).reshape(-1) + (B - 1) / 2.0
            b = torch.floor(u)
            f = u - b
            b = b.long()
            row = torch.zeros((B + 1, N), device=DEV, dtype=torch.float64)
            row.index_add_(0, b, (flat * (1.0 - f)).T)
            row.index_add_(0, b + 1, (flat * f).T)
            out[:, k] = row[:B].T
    else:
        # slice samples by direct sums, the angles theta and pi - theta from
        # one product (their first frequencies differ in sign only)
        nj = B // 2 + 1
        j = torch.arange(nj, device=DEV, dtype=torch.float64)
        ks = torch.arange(nh // 2 + 1, device=DEV)
        t1 = (j[None] / B * co[ks][:, None]).reshape(-1)
        t2 = (j[None] / B * si[ks][:, None]).reshape(-1)
        ph1, ph2 = 2.0 * math.pi * x[:, None] * t1[None], 2.0 * math.pi * x[:, None] * t2[None]
        E1 = torch.cat([torch.cos(ph1), torch.sin(ph1)], 1)  # [L][2T]
        c2, s2 = torch.cos(ph2), torch.sin(ph2)              # [L][T]
        T = t1.numel()
        amp = torch.sinc(t1) * torch.sinc(t2)
        sb = torch.arange(B, device=DEV, dtype=torch.float64) - (B - 1) / 2.0
        w = torch.full((nj,), 2.0, device=DEV, dtype=torch.float64)
        w[0] = w[-1] = 1.0
        kern = 2.0 * math.pi * j[:, None] * sb[None] / B
        Cb, Sb = torch.cos(kern) * w[:, None] / B, torch.sin(kern) * w[:, None] / B
        # j = -B/2 is the one unpaired frequency: its real part
        step = max(1, int(2e9 / (16.0 * L * T)))
        for i in range(0, N, step):
            m = min(step, N - i)
            a = (img[i:i + m].reshape(m * L, L) @ E1).reshape(m, L, 2 * T)
            A, Bs = a[:, :, :T], a[:, :, T:]
            cc, ss = (A * c2).sum(1), (Bs * s2).sum(1)
            cs, sc = (A * s2).sum(1), (Bs * c2).sum(1)
            for sign in (1.0, -1.0):
                re = ((cc - sign * ss) * amp).reshape(m, -1, nj)
                im = (-(cs + sign * sc) * amp).reshape(m, -1, nj)
                rows = re @ Cb - im @ Sb
                if sign > 0:
                    out[i:i + m, :nh // 2 + 1] = rows[:, :min(nh, nh // 2 + 1)]
                else:
                    for k in range(1, nh // 2 + 1):
                        if nh - k > nh // 2:
                            out[i:i + m, nh - k] = rows[:, k]
        if case["metric"] != "rfsw2":
            out.clamp_(min=0.0)
    return torch.cat([out, out.flip(2)], 1)


def _quantiles64(rows, L, M, case):
    """Quantiles [N][parts][n][M] of rows [N][n][B]."""
    B, h = rows.shape[-1], 2.0 / L
    if case["metric"] == "rfsw2":
        j = torch.arange(B // 2 + 1, device=DEV, dtype=torch.float64)
        f = torch.fft.irfft(torch.fft.rfft(rows) * j, n=B)
        U = torch.stack([f.clamp(min=0.0), (-f).clamp(min=0.0)], 1)
    else:
        U = rows[:, None]
    F = torch.cumsum(U, -1)
    p = torch.arange(M, device=DEV, dtype=torch.float64)
    z = p / M if case["level_rule"] else (p + 0.5) / M
    tau = (z * F[..., -1:]).contiguous()
    idx = torch.searchsorted(F.contiguous(), tau).clamp(max=B - 1)
    Fp = torch.cat([torch.zeros_like(F[..., :1]), F[..., :-1]], -1).gather(-1, idx)
    u = U.gather(-1, idx)
    frac = torch.where(u > 0, (tau - Fp) / u, torch.zeros_like(u)).clamp(0.0, 1.0)
    q = (idx.double() - B / 2.0 + frac) * h
    return torch.where(tau == 0, torch.full_like(q, -0.5 * B * h), q)


def _center64(q):
    n = q.shape[2]
    th = 2.0 * math.pi * torch.arange(n, device=DEV, dtype=torch.float64) / n
    e = torch.stack([torch.cos(th), torch.sin(th)], 1)
    a = (2.0 / n) * torch.einsum("ipk,kd->ipd", q.mean(-1), e)
    return a, q - torch.einsum("ipd,kd->ipk", a, e)[..., None], e


def _quant_of(img, L, n, M, case, chunk):
    B = swalign.bins_of(_params(case, L, M))
    return torch.cat([_quantiles64(_rows64(img[i:i + chunk].double(), L, n, B, case), L, M, case)
                      for i in range(0, img.shape[0], chunk)])


def _curves64(uq, ut, L, case):
    """D [Nq][Nt][n] and shifts [Nq][Nt][n][2]."""
    Nq, parts, n, M = uq.shape
    aq, cq, e = _center64(uq)
    at, ct, _ = _center64(ut)
    rot = torch.stack([torch.stack([e[:, 0], -e[:, 1]], 1), e.flip(1)], 1)  # [n][2][2]
    c = aq[:, None, :, None] - torch.einsum("lde,jpe->jpld", rot, at)[None]  # [Nq][Nt][parts][n][2]
    if case["metric"] == "msw2":
        fq, ft = (cq, ct) if case["translation"] else (uq, ut)
        k = torch.arange(n, device=DEV)
        roll = (k[None, :] - k[:, None]) % n  # [l][k]
        D = torch.empty((Nq, ut.shape[0], n), device=DEV, dtype=torch.float64)
        for j in range(ut.shape[0]):
            g = (fq[:, 0].square().sum(-1)[:, :, None] + ft[j, 0].square().sum(-1)[None, None, :]
                 - 2.0 * fq[:, 0] @ ft[j, 0].T)  # [Nq][k][k']
            D[:, j] = g[:, k[None, :], roll].amax(-1) / M
        s = c[:, :, 0]
        return D, s if case["translation"] else torch.zeros_like(s)
    X = torch.fft.rfft(cq, dim=2).permute(1, 2, 0, 3)  # [parts][f][Nq][M]
    Y = torch.fft.rfft(ct, dim=2).permute(1, 2, 3, 0).conj()
    C = sum(X[p] @ Y[p] for p in range(parts))
    corr = torch.fft.irfft(C.permute(1, 2, 0), n=n)
    D = cq.square().sum((1, 2, 3))[:, None, None] + ct.square().sum((1, 2, 3))[None, :, None]
    D = (D - 2.0 * corr) / (n * M)
    rho, s = 0.5, c[:, :, 0]
    if parts == 2:
        d = c[:, :, 0] - c[:, :, 1]
        D = D + 0.25 * d.square().sum(-1)
        rho, s = 1.0, 0.5 * (c[:, :, 0] + c[:, :, 1])
    if not case["translation"]:
        D, s = D + rho * s.square().sum(-1), torch.zeros_like(s)
    elif case["shift_grid"]:
        K, step = case["shift_grid"], 8 * (2.0 / L) / 16.0
        gp = torch.round(s / step).clamp(-K, K) * step
        D, s = D + rho * (s - gp).square().sum(-1), gp
    return D, s


def _best64(uq, ut, L, case):
    """The doubles (shift, d2) of every result, [rows][3]."""
    per = max(1, int(2e8 / (ut.shape[0] * uq.shape[2])))
    out = []
    for i in range(0, uq.shape[0], per):
        D, s = _curves64(uq[i:i + per], ut, L, case)
        d, l = D.min(-1)
        r = torch.cat([s.gather(2, l[..., None, None].expand(*l.shape, 1, 2))[:, :, 0],
                       d[..., None]], -1)
        if case["mode"] == 1:
            j = d.argmin(1)
            r = r[torch.arange(r.shape[0], device=DEV), j][:, None]
        out.append(r.reshape(-1, 3))
    return torch.cat(out)


def exact(case, seed):
    if case["projector"] == "slice":
        flops = sum((Nq + Nt) * 2.0 * L * L * (case["n"] / 2) *
                    swalign.bins_of(_params(case, L, M)) / 2
                    for L, _, M, Nq, Nt in _sizes(case))
        if flops > 1e13:
            return None
    ins = _inputs(case, seed)
    if case["kind"] != "uneven":
        ins = {case["L"]: ins}
    res = {}
    for L, q_L, M, Nq, Nt in _sizes(case):
        q, t = ins[L]
        if q_L != L:
            q = 0.25 * q.repeat_interleave(2, 1).repeat_interleave(2, 2)
        chunk = max(1, int(1e9 / (8.0 * L * L + 40.0 * case["n"] * M)))
        n = case["n"]
        if case["kind"] == "stages":
            B = swalign.bins_of(_params(case, L, M))
            rows = _rows64(q.double(), L, n, B, case)
            u = _quantiles64(rows, L, M, case)
            a, cu, _ = _center64(u)
            v = {"rows": rows, "scale": 1.0 / q.double().clamp(min=0.0).sum((1, 2)),
                 "quantiles": u, "center": a, "norm": cu.square().sum((2, 3))}
            if case["metric"] != "rfsw2":
                v = {k: x[:, 0] if k in ("quantiles", "center", "norm") else x
                     for k, x in v.items()}
            return v
        uq, ut = _quant_of(q, L, n, M, case, chunk), _quant_of(t, L, n, M, case, chunk)
        if case["kind"] == "pair":
            D, s = _curves64(uq, ut, L, case)
            d, l = D[0, 0].min(0)
            return {"curve": D[0, 0], "shifts": s[0, 0],
                    "best": (None, torch.cat([s[0, 0, l], d[None]])[None])}
        res[str(L)] = (None, _best64(uq, ut, L, case))
    return res if case["kind"] == "uneven" else res[str(case["L"])]
