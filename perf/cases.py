"""What the library is asked to do in real use, as cases that can be timed and compared.

Each case goes through the package's public calls (``ginterp.compress`` / ``decompress``,
their forms on kept buffers, ``Batch``, the Huffman stage, the quality report).  Sizes
are those of the repository's benchmark and tests: the 64^3 field of the smoke test, the
512^3 density field, the uneven batch, the cubes of the request stream (32 .. 512 per
edge), the 1024^3 outlier-heavy field and the 512 MiB 1-D / 2-D fields.  Fields are drawn
on the GPU from the seed with the statistics of ``fields.py``: Gaussian random fields of
a power-law spectrum, exp of one (density-like), plane sine waves with noise, and
piecewise-smooth fields with steps.

A case's ``do`` says which calls one pass makes:
  roundtrip  compress() and decompress(), which allocate their results and check the
             outlier count: the calls of the README
  cycle      compress_into() and decompress_into() on kept buffers: a solver that keeps
             its time steps compressed
  compress, decompress   one of the two, on kept buffers
  batch      Batch.round_trip(): several fields in one call per direction
  encode, decode         the Huffman stage on a field's quant-codes, on kept buffers
  quality    quality(): entropy, nonzero codes, PSNR of a field and its reconstruction
"""
from __future__ import annotations

import math

import torch

from paper_2312_05492_gb300 import ginterp as G

DEV = "cuda"


def listed():
    return [
        # the smallest call: one small field, linear, fixed order (latency and launches)
        dict(name="roundtrip_grf_64", do="roundtrip", field="grf", beta=3.0, nz=64, ny=64, nx=64, eb=1e-3,
             order="012", levels="000", cubic="000", auto=False, ndim=3, domain=8),
        # the headline field, one direction at a time: post-processing reads what a run wrote
        dict(name="compress_density_512", do="compress", field="lognormal", beta=11 / 3, nz=512, ny=512, nx=512,
             eb=1e-3, auto=True, ndim=3, domain=8),
        dict(name="decompress_density_512", do="decompress", field="lognormal", beta=11 / 3, nz=512, ny=512,
             nx=512, eb=1e-3, auto=True, ndim=3, domain=8),
        # rows that are odd and not 16-byte aligned, splines at every level, an untuned configuration
        dict(name="roundtrip_waves_ragged", do="roundtrip", field="sines", beta=0.0, nz=449, ny=449, nx=235,
             eb=1e-3, order="102", levels="111", cubic="000", auto=False, ndim=3, domain=8),
        # three uneven anisotropic fields with their own bounds in one call
        dict(name="batch_uneven", do="batch", cubes=False, count=3, lo=0, hi=0, sizes=0),
        # what the serving loop packs together: eight cubes of its edge range
        dict(name="batch_requests", do="batch", cubes=True, count=8, lo=32, hi=256, sizes=7),
        # the largest field, outlier-heavy at a tight bound
        dict(name="cycle_shocks_1024", do="cycle", field="shocks", beta=3.0, nz=1024, ny=1024, nx=1024, eb=1e-5,
             order="012", levels="111", cubic="000", auto=False, ndim=3, domain=8),
        # a stack of 2-D slices (16^2 chunks) and a set of 1-D series (512-point chunks)
        dict(name="cycle_slices_2d", do="cycle", field="grf", beta=3.0, nz=32, ny=2048, nx=2048, eb=1e-3, auto=True,
             ndim=2, domain=8),
        dict(name="cycle_series_1d", do="cycle", field="grf", beta=3.0, nz=1, ny=64, nx=1 << 21, eb=1e-3, auto=True,
             ndim=1, domain=8),
        # the lossless stage on the headline field's codes, one codebook kept over time steps
        dict(name="encode_density_512", do="encode", field="lognormal", beta=11 / 3, nz=512, ny=512, nx=512, eb=1e-3,
             auto=True, ndim=3, domain=8),
        dict(name="decode_density_512", do="decode", field="lognormal", beta=11 / 3, nz=512, ny=512, nx=512, eb=1e-3,
             auto=True, ndim=3, domain=8),
        # the report read when a bound is chosen
        dict(name="quality_density_384", do="quality", field="lognormal", beta=11 / 3, nz=384, ny=384, nx=384,
             eb=1e-3, auto=True, ndim=3, domain=8),
    ]


def draw(rng):
    do = rng.choice(["roundtrip", "cycle", "compress", "decompress", "batch", "encode", "decode", "cycle2", "cycle1",
                     "quality"])
    if do == "batch":
        hi = int(round(math.exp(rng.uniform(math.log(64), math.log(320)))))
        return dict(do="batch", cubes=True, count=rng.randint(2, 8), lo=32, hi=hi, sizes=rng.randrange(1 << 30))
    ndim = {"cycle2": 2, "cycle1": 1}.get(do, 3)
    n = math.exp(rng.uniform(math.log(3e4), math.log(1.3e8)))
    if ndim == 3:
        a, b = math.exp(rng.uniform(-0.7, 0.7)), math.exp(rng.uniform(-0.7, 0.7))
        e = n ** (1 / 3)
        nz, ny, nx = (max(17, int(v)) for v in (e * a, e * b, e / (a * b)))
    elif ndim == 2:
        nz = rng.choice([1, 1, 3, 8, 32])
        a = math.exp(rng.uniform(-0.7, 0.7))
        e = math.sqrt(n / nz)
        ny, nx = max(33, int(e * a)), max(33, int(e / a))
    else:
        nz, ny = 1, rng.choice([1, 7, 64])
        nx = max(600, int(n / ny))
    if rng.random() < 0.5:  # rows of whole 32-byte sectors; the others as they come, odd ones among them
        nx = max(32, nx // 32 * 32)
    auto = rng.random() < 0.5
    c = dict(do={"cycle2": "cycle", "cycle1": "cycle"}.get(do, do), field=rng.choice(["grf", "lognormal", "sines", "shocks"]),
             beta=rng.choice([5 / 3, 3.0, 11 / 3, 4.0]), nz=nz, ny=ny, nx=nx, eb=rng.choice([1e-2, 1e-3, 1e-4]), auto=auto,
             ndim=ndim, domain=rng.choice([8, 8, 32]) if ndim == 3 and do in ("roundtrip", "cycle") else 8)
    if not auto:
        c.update(order=rng.choice(["012", "021", "102", "120", "201", "210"]),
                 levels=rng.choice(["000", "111", "011", "111"]), cubic=rng.choice(["000", "111", "010"]))
    return c


# ------------------------------------------------------------------ inputs
def _grf(shape, beta, gen, ndim=3):
    """Gaussian random field, spectrum ~ |k|^-beta over the last ndim axes, mean 0, std 1."""
    axes = tuple(range(3 - ndim, 3))
    spec = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV), dim=axes)
    k2 = torch.zeros((1, 1, 1), device=DEV)
    for a in axes:
        f = torch.fft.rfftfreq(shape[a], device=DEV) if a == 2 else torch.fft.fftfreq(shape[a], device=DEV)
        k2 = k2 + f.reshape([-1 if b == a else 1 for b in range(3)]) ** 2
    spec *= torch.where(k2 > 0, k2.clamp_min(1e-30) ** (-beta / 4), torch.zeros_like(k2))
    f = torch.fft.irfftn(spec, s=[shape[a] for a in axes], dim=axes)
    del spec
    f -= f.mean()
    f /= f.std().clamp_min(1e-20)
    return f.contiguous()


def _sines(shape, gen, cpu):
    f = torch.zeros(shape, device=DEV)
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) / n for n in shape]
    kv = torch.randint(-16, 17, (32, 3), generator=cpu)
    amp = 0.5 + 0.5 * torch.rand(32, generator=cpu)
    ph = 2 * math.pi * torch.rand(32, generator=cpu)
    for w in range(32):
        t = [(2 * math.pi * float(kv[w, a])) * ax[a] for a in range(3)]
        t = (t[0][:, None, None] + (t[1][None, :, None] + float(ph[w]))).float() + t[2][None, None, :].float()
        f += float(amp[w]) * torch.sin(t)
    f += (0.01 * f.std()) * torch.randn(shape, generator=gen, device=DEV)
    return f.contiguous()


def _shocks(shape, beta, gen, cpu, ndim):
    f = _grf(shape, beta, gen, ndim)
    for _ in range(8):
        nrm = torch.randn(3, generator=cpu, dtype=torch.float64)
        nrm /= nrm.norm()
        c = float((nrm * torch.rand(3, generator=cpu, dtype=torch.float64) * torch.tensor(shape)).sum())
        sign = 10.0 if float(torch.rand(1, generator=cpu)) < 0.5 else -10.0
        zy = (float(nrm[0]) * torch.arange(shape[0], device=DEV)[:, None, None]
              + float(nrm[1]) * torch.arange(shape[1], device=DEV)[None, :, None])
        x = float(nrm[2]) * torch.arange(shape[2], device=DEV)[None, None, :]
        f += torch.where(x > c - zy, sign, 0.0)
    return f.contiguous()


def _field(kind, beta, shape, seed, ndim=3):
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    cpu = torch.Generator().manual_seed(int(seed))
    if kind == "sines":
        return _sines(shape, gen, cpu)
    if kind == "shocks":
        return _shocks(shape, beta, gen, cpu, ndim)
    f = _grf(shape, beta, gen, ndim)
    return torch.exp(f).contiguous() if kind == "lognormal" else f


def _digits(s):
    return tuple(int(v) for v in s)


def _config(c):
    cfg = G.Config(autotune=bool(c["auto"]), ndim=c["ndim"], domain_x=c["domain"])
    if not c["auto"]:
        cfg.dim_order, cfg.level_kind, cfg.cubic_kind = _digits(c["order"]), _digits(c["levels"]), _digits(c["cubic"])
    return cfg


def _kept(x, cfg, capacity):
    """Buffers that a program keeps from call to call (the unused end of the outlier list holds zeros)."""
    bufs = G.allocate(tuple(x.shape), cfg, x.device, capacity=capacity)
    bufs["out_idx"].zero_()
    bufs["out_val"].zero_()
    cf = G.CompressedField(tuple(x.shape), cfg, bufs["header"], bufs["anchors"], bufs["codes"], bufs["out_idx"],
                           bufs["out_val"], bufs["hist"], bufs["capacity"])
    ws = torch.empty(G.interp_workspace_bytes(tuple(x.shape), cfg.to_c()), dtype=torch.uint8, device=x.device)
    return bufs, cf, ws


def _batch_fields(c, seed):
    if not c["cubes"]:
        return [("grf", 4.0, (100, 500, 500), 1e-2), ("grf", 5 / 3, (256, 384, 384), 1e-3),
                ("sines", 0.0, (449, 449, 235), 1e-4)]
    g = torch.Generator().manual_seed(int(c["sizes"]))
    got = []
    for _ in range(c["count"]):
        u = float(torch.rand(1, generator=g))
        e = int(round(math.exp(math.log(c["lo"]) + u * (math.log(c["hi"]) - math.log(c["lo"])))))
        got.append(("grf", 3.0, (e, e, e), (1e-2, 1e-3, 1e-4)[int(torch.randint(3, (1,), generator=g))]))
    return got


def prepare(case, seed):
    c, do = case, case["do"]
    if do == "batch":
        fs = _batch_fields(c, seed)
        xs = [_field(k, b, s, seed * 16 + i) for i, (k, b, s, _) in enumerate(fs)]
        cfgs = [G.Config(autotune=True) for _ in fs]
        # the serving loop's outlier room: one entry for every 16 points
        b = G.Batch(xs, [f[3] for f in fs], cfgs, capacities=[max(1024, x.numel() // 16) for x in xs])
        for buf in b.bufs:
            buf["out_idx"].zero_()
            buf["out_val"].zero_()
        return dict(do=do, batch=b)
    x = _field(c["field"], c["beta"], (c["nz"], c["ny"], c["nx"]), seed, c["ndim"])
    cfg = _config(c)
    if do == "roundtrip":
        return dict(do=do, x=x, eb=c["eb"], cfg=cfg)
    if do == "quality":
        cf = G.compress(x, c["eb"], cfg)
        return dict(do=do, x=x, cf=cf, xr=G.decompress(cf))
    bufs, cf, ws = _kept(x, cfg, x.numel() // 4 + 1024)
    st = dict(do=do, x=x, eb=c["eb"], cfg=cfg, bufs=bufs, cf=cf, ws=ws)
    if do in ("cycle", "decompress"):
        st["out"] = torch.empty_like(x)
    if do in ("decompress", "encode", "decode"):
        G.compress_into(x, c["eb"], cfg, bufs, ws)
    if do in ("encode", "decode"):
        lengths, codewords = G.huffman_codebook(bufs["hist"], cfg.radius)
        st["hs"] = G.huffman_encode(bufs["codes"], cfg.radius, lengths, codewords)
        if do == "encode":
            st["hs"].words.zero_()
        else:
            st["codes"] = torch.empty_like(bufs["codes"])
    return st


# ------------------------------------------------------------------ one pass
def _parts(b):
    return {k: b[k] for k in ("codes", "anchors", "out_idx", "out_val", "hist", "header")}


def run(st):
    do = st["do"]
    if do == "roundtrip":
        cf = G.compress(st["x"], st["eb"], st["cfg"])
        xr = G.decompress(cf)
        # the outliers are the points of code 0, whose values xrec holds (compress() has read their number)
        return dict(codes=cf.codes, anchors=cf.anchors, hist=cf.hist, header=cf.header, n_outliers=cf.n_outliers, xrec=xr)
    if do == "batch":
        b = st["batch"]
        b.round_trip()
        return [dict(_parts(buf), xrec=o) for buf, o in zip(b.bufs, b.outs)]
    if do == "quality":
        return G.quality(st["cf"], st["x"], st["xr"])
    if do == "encode":
        hs = G.huffman_reencode(st["hs"], st["bufs"]["codes"])
        return dict(offsets=hs.offsets, words=hs.words)
    if do == "decode":
        return G.huffman_decode(st["hs"], st["codes"])
    if do in ("cycle", "compress"):
        G.compress_into(st["x"], st["eb"], st["cfg"], st["bufs"], st["ws"])
    if do in ("cycle", "decompress"):
        G.decompress_into(st["cf"], st["out"])
    return {"cycle": lambda: dict(_parts(st["bufs"]), xrec=st["out"]), "compress": lambda: _parts(st["bufs"]),
            "decompress": lambda: st["out"]}[do]()


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c, do = case, case["do"]
    if do == "batch":
        n = sum(math.prod(f[2]) for f in _batch_fields(c, 0))
        return dict(bytes=12.1 * n, flops=40.0 * n)
    n = c["nz"] * c["ny"] * c["nx"]
    anchors = n / {3: 512, 2: 256, 1: 512}[c["ndim"]]
    if do in ("encode", "decode"):  # 16-bit codes on one side, about 2.3 bits a code on the other (at a bound of 1e-3)
        return dict(bytes=2.3 * n, flops=4.0 * n)
    if do == "quality":
        return dict(bytes=8.0 * n, flops=6.0 * n)
    one = 6.0 * n + 4.0 * anchors  # values on one side, codes and anchors on the other; about 20 operations a point
    both = do in ("roundtrip", "cycle")
    return dict(bytes=one * (2 if both else 1), flops=20.0 * n * (2 if both else 1))


# ------------------------------------------------------------------ the same in 64 bits
def _replay64(dims, codes, anchors, out_idx, out_val, h):
    """The field that codes, anchors and outliers stand for (8^3 chunks), in plain float64."""
    order, R = list(h.cfg.dim_order), h.cfg.radius
    q = codes.to(torch.int32).bitwise_and_(0xFFFF).reshape(dims)
    v = torch.zeros(dims, dtype=torch.float64, device=codes.device)
    v[::8, ::8, ::8] = anchors.reshape(v[::8, ::8, ::8].shape).double()
    kept = torch.zeros(math.prod(dims), dtype=torch.float64, device=codes.device)
    kept[out_idx.to(torch.int64).bitwise_and_(0xFFFFFFFF)] = out_val.double()
    kept = kept.reshape(dims)
    for lvl, s in ((2, 4), (1, 2), (0, 1)):
        twoe = 2.0 * h.eb_abs / h.alpha ** lvl
        for k, d in enumerate(order):
            sl = [slice(None, None, s if a in order[:k] else 2 * s) for a in range(3)]
            sl[d] = slice(None)
            grid = v[tuple(sl)]
            n = torch.arange(s, dims[d], 2 * s, device=v.device)
            if not n.numel():
                continue
            lo = n // 8 * 8
            hi = (lo + 8).clamp_max(dims[d] - 1)
            shape = [-1 if a == d else 1 for a in range(3)]
            has = {o: ((n + o >= lo) & (n + o <= hi)).reshape(shape) for o in (-3 * s, s, 3 * s)}
            at = {o: grid.index_select(d, (n + o).clamp(0, dims[d] - 1)) for o in (-3 * s, -s, s, 3 * s)}
            m3, m1, p1, p3 = at[-3 * s], at[-s], at[s], at[3 * s]
            p = (m1 + p1) / 2
            if h.cfg.level_kind[lvl]:
                p = torch.where(has[3 * s], (3 * m1 + 6 * p1 - p3) / 8, p)
                p = torch.where(has[-3 * s], (6 * m1 - m3 + 3 * p1) / 8, p)
                cubic = (23 * (m1 + p1) - 3 * (m3 + p3)) / 40 if h.cfg.cubic_kind[d] else (9 * (m1 + p1) - (m3 + p3)) / 16
                p = torch.where(has[-3 * s] & has[3 * s], cubic, p)
            p = torch.where(has[s], p, m1)
            sl[d] = slice(s, None, 2 * s)
            c = q[tuple(sl)]
            v[tuple(sl)] = torch.where(c == 0, kept[tuple(sl)], p + (c - R).double() * twoe)
    return v


def _anchors64(x, ndim):
    a = {3: 8, 2: 16, 1: 512}[ndim]
    return x[tuple(slice(None, None, a if ax >= 3 - ndim else 1) for ax in range(3))].double().reshape(-1)


def exact(case, seed):
    c, do = case, case["do"]
    st = prepare(c, seed)
    if do == "decompress":
        cf = st["cf"]
        h = cf.host_header()
        n = int(h.n_outliers)
        return _replay64(cf.dims, cf.codes, cf.anchors, cf.out_idx[:n], cf.out_val[:n], h)
    if do == "quality":
        x, xr = st["x"].double().reshape(-1), st["xr"].double().reshape(-1)
        h = st["cf"].hist.double()
        p = h[h > 0] / h.sum()
        err = x - xr
        sse, vmin, vmax = float(err.square().sum()), float(x.min()), float(x.max())
        return dict(entropy_bits=float(-(p * p.log2()).sum()), sse=sse, max_abs_err=float(err.abs().max()), vmin=vmin,
                    vmax=vmax, psnr_db=20 * math.log10(vmax - vmin) - 10 * math.log10(sse / x.numel()))
    if do == "batch":  # whole numbers but for the anchors; the reconstruction follows from the codes of the same pass
        return [dict(codes=None, anchors=_anchors64(x, 3)) for x in st["batch"].xs]
    if do in ("roundtrip", "cycle", "compress"):
        return dict(codes=None, anchors=_anchors64(st["x"], c["ndim"]))
    return None
