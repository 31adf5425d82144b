"""The work this package is used for, as cases whose time is measured.

Each case goes through the public entry points of paper_2308_11759_gb300 as a
program that uses it would.  The kinds:

  compress    a field arrives on the device: its tolerance schedule from its
              range, then all components (the simulation writing a step)
  roundtrip   the same, and reconstructions from the streams
  retrieve    one reconstruction of a whole field at a tolerance
  sweep       progressive access: the first component, then refinement in
              place, one component at a time
  box         one sub-box of a resident field at a tolerance
  boxes       a list of sub-boxes of resident fields in one call
  batch       the many uneven fields of one time step through a kept plan, and
              all of them read back
  serve       a burst of sub-box queries to the progressive-query server
  checkpoint  streams to host bytes and back
  derivative  the derivatives of a velocity field (vorticity, w_zz)

Fields are made on the GPU from the seed alone: random-phase k^-5/3 fields,
sums of Gaussians with a little noise, and k^-5/3 fields with sharp fronts.
"""
import math
import random

import numpy as np
import torch

import paper_2308_11759_gb300 as pcz

_T = {"f32": torch.float32, "f64": torch.float64}

# ---- the cases -------------------------------------------------------------------


def listed():
    return [
        # a large simulation field written once: 8 decades of tolerance (the
        # large plain-method configuration)
        dict(name="compress_f32_512", kind="compress", dtype="f32", nz=512, ny=512, nx=512, n=8, schedule="decade",
             field="powerlaw"),
        # a near-lossless archive of a double-precision field with sharp
        # fronts, 12 decades (the 1024^3 configuration's method, on the shape
        # of Table 1's Miranda field)
        dict(name="compress_f64_fronts", kind="compress", dtype="f64", nz=256, ny=384, nx=384, n=12,
             schedule="decade", field="fronts"),
        # the smallest configuration: a 64^3 field coded and read back at every
        # k, where launches and host latency count
        dict(name="roundtrip_f64_64", kind="roundtrip", dtype="f64", ndims=3, nz=64, ny=64, nx=64, n=4,
             schedule="binary", field="gaussians", all_k=True),
        # a 2D slice or surface field of odd extents, coded and read back
        dict(name="roundtrip_f32_2d", kind="roundtrip", dtype="f32", ndims=2, nz=1, ny=2311, nx=3001, n=6,
             schedule="decade", field="powerlaw", all_k=False),
        # a whole large field at one mid tolerance, for analysis
        dict(name="retrieve_f32_512", kind="retrieve", dtype="f32", nz=512, ny=512, nx=512, n=8, k=6,
             schedule="decade", field="powerlaw"),
        # progressive refinement of a double-precision field of odd extents
        dict(name="sweep_f64_odd", kind="sweep", dtype="f64", nz=251, ny=379, nx=381, n=8, k=8, schedule="decade",
             field="powerlaw"),
        # a visualisation client asks for one region at a modest tolerance
        dict(name="box_f32_64", kind="box", dtype="f32", size=256, side=64, n=8, k=4),
        # an analysis pass over 64 regions of two resident fields
        dict(name="boxes_f64", kind="boxes", dtype="f64", size=256, fields=2, count=64, boxes=1, low=8, high=128,
             n=8),
        # the uneven batch of one time step: 64 fields, half 2D and half 3D
        dict(name="batch_f32_64", kind="batch", dtype="f32", count=64, n=6, shapes=3),
        # 128 queries arriving together at the server of 16 fields
        dict(name="serve_f32", kind="serve", dtype="f32", size=256, fields=16, count=128, boxes=2, n=8),
        # checkpoint and restart of one compressed field
        dict(name="checkpoint_f32", kind="checkpoint", dtype="f32", nz=128, ny=128, nx=128, n=8, schedule="decade",
             field="powerlaw"),
        # the use case's derivatives on a velocity field of Miranda's shape
        dict(name="derivative_f64", kind="derivative", dtype="f64", nz=256, ny=384, nx=384, h=1.0),
    ]


_MOST = {"f32": 512 ** 3, "f64": 256 * 384 * 384}  # values of the largest fields


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _shape(rng, most, ndims=3, least=32 ** 3):
    """Extents of a field of up to `most` values, the size spread over its logarithm; odd extents as they come."""
    side = _log(rng, least, most / 2.5) ** (1.0 / ndims)
    ext = [max(8, int(side * math.exp(rng.uniform(-0.3, 0.3)))) for _ in range(ndims)]
    return [1] * (3 - ndims) + ext


def draw(rng: random.Random):
    kind = rng.choice(["compress", "compress", "roundtrip", "roundtrip", "retrieve", "retrieve", "sweep", "box",
                       "boxes", "batch", "serve", "checkpoint", "derivative"])
    dt = rng.choice(["f32", "f64"])
    n = rng.randint(2, 8) if dt == "f32" else rng.randint(2, 12)
    schedule = rng.choice(["decade", "decade", "binary"])
    field = rng.choice(["powerlaw", "powerlaw", "gaussians", "fronts"])
    c = dict(kind=kind, dtype=dt)
    if kind in ("compress", "retrieve", "sweep"):
        nz, ny, nx = _shape(rng, _MOST[dt])
        c.update(nz=nz, ny=ny, nx=nx, n=n, schedule=schedule, field=field)
        if kind != "compress":
            c.update(k=rng.randint(1, n))
    elif kind == "roundtrip":
        nd = rng.choice([1, 2, 2, 3])
        nz, ny, nx = _shape(rng, 4 * 10 ** 6 if nd == 1 else 16 * 10 ** 6, nd, 4096)
        c.update(ndims=nd, nz=nz, ny=ny, nx=nx, n=min(n, 6), schedule=schedule, field="powerlaw" if nd < 3 else field,
                 all_k=rng.random() < 0.5)
    elif kind == "box":
        size = rng.randint(96, 256)
        c.update(size=size, side=min(size, int(_log(rng, 8, 200))), n=n, k=rng.randint(1, n))
    elif kind == "boxes":
        c.update(size=rng.randint(128, 256), fields=rng.randint(1, 4), count=int(_log(rng, 4, 128)),
                 boxes=rng.randint(3, 10 ** 6), low=8, high=rng.choice([32, 64, 128]), n=n)
    elif kind == "batch":
        c.update(count=int(_log(rng, 4, 64 if dt == "f32" else 24)), n=min(n, 6), shapes=rng.randint(4, 10 ** 6))
    elif kind == "serve":
        c.update(size=4 * rng.randint(24, 64), fields=rng.randint(2, 16 if dt == "f32" else 6),
                 count=int(_log(rng, 8, 128)), boxes=rng.randint(3, 10 ** 6), n=n)
    elif kind == "checkpoint":
        nz, ny, nx = _shape(rng, 160 ** 3)
        c.update(nz=nz, ny=ny, nx=nx, n=n, schedule=schedule, field=field)
    else:
        nz, ny, nx = _shape(rng, 256 * 384 * 384)
        c.update(nz=nz, ny=ny, nx=nx, h=rng.choice([1.0, 0.5, 2.0 * math.pi / nx]))
    return c


# ---- fields ----------------------------------------------------------------------


def _rand_state(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFFFFFF)
    return g


def _powerlaw(shape, g, dtype):
    """A random-phase Gaussian field with P(k) ~ k^-5/3 and unit variance."""
    freqs = [torch.fft.fftfreq(s, device="cuda", dtype=dtype) for s in shape[:-1]]
    freqs.append(torch.fft.rfftfreq(shape[-1], device="cuda", dtype=dtype))
    k2 = sum(f.reshape([-1 if a == b else 1 for b in range(len(shape))]) ** 2 for a, f in enumerate(freqs))
    k2.view(-1)[0] = 1.0
    amp = k2.pow_(-5.0 / 12.0)
    amp.view(-1)[0] = 0.0
    phase = torch.rand(amp.shape, generator=g, device="cuda", dtype=dtype).mul_(2.0 * math.pi)
    f = torch.fft.irfftn(torch.polar(amp, phase), s=shape)
    f -= f.mean()
    f /= f.std()
    return f


def _axis(n, a, nd, dtype):
    return torch.arange(n, device="cuda", dtype=dtype).reshape([-1 if a == b else 1 for b in range(nd)])


def _gaussians(shape, g, r, dtype):
    """A sum of 32 anisotropic Gaussians and noise of 1e-3."""
    out = torch.randn(shape, generator=g, device="cuda", dtype=dtype).mul_(1e-3)
    nd = len(shape)
    for _ in range(32):
        p = None
        for a, s in enumerate(shape):
            q = torch.exp(-0.5 * ((_axis(s, a, nd, dtype) - r.uniform(0, s)) / r.uniform(2.0, 16.0)) ** 2)
            p = q if p is None else p * q
        out.add_(p, alpha=r.uniform(-1.0, 1.0))
    return out


def _fronts(shape, g, r, dtype):
    """A k^-5/3 field with 24 sharp tanh interfaces."""
    out = _powerlaw(shape, g, dtype)
    nd = len(shape)
    ax = [_axis(s, a, nd, dtype) for a, s in enumerate(shape)]
    for j in range(24):
        amp = r.uniform(-2.0, 2.0)
        if j % 2 == 0:
            nrm = [r.gauss(0.0, 1.0) for _ in shape]
            ln = math.sqrt(sum(v * v for v in nrm)) or 1.0
            d = sum(x * (v / ln) for x, v in zip(ax, nrm))
            d = d - sum(r.uniform(0, s) * (v / ln) for s, v in zip(shape, nrm))
        else:
            rad = r.uniform(0.05, 0.3) * min(shape)
            d = torch.sqrt(sum((x - r.uniform(0, s)) ** 2 for x, s in zip(ax, shape))) - rad
        out.add_(torch.tanh(d), alpha=amp)
    return out


def _field(kind, shape, dt, seed):
    g, r = _rand_state(seed), random.Random(int(seed))
    dtype = _T[dt]
    if kind == "powerlaw":
        return _powerlaw(tuple(shape), g, dtype).contiguous()
    if kind == "gaussians":
        return _gaussians(tuple(shape), g, r, dtype).contiguous()
    return _fronts(tuple(shape), g, r, dtype).contiguous()


def _schedule(x, case):
    if case["schedule"] == "binary":
        return pcz.field_tau_schedule(x, "binary", case["n"], param=4)
    return pcz.field_tau_schedule(x, "decade", case["n"], param=1 if case["n"] > 8 else 2)


def _shape_of(case):
    nd = case.get("ndims", 3)
    return [case["nz"], case["ny"], case["nx"]][3 - nd:]


def _batch_shapes(count, seed):
    """Half 2D with extents in [256, 4096], half 3D between 32^3 and 256 x 384 x 384."""
    r = random.Random(seed)
    out = []
    for i in range(count):
        if i % 2 == 0:
            out.append((r.randint(256, 4096), r.randint(256, 4096)))
        else:
            out.append((r.randint(32, 256), r.randint(32, 384), r.randint(32, 384)))
    return out


def _sides(case, low, high, align):
    """The sub-boxes' extents, log-uniform in [low, high]: the case's own."""
    r = random.Random(case["boxes"])
    return [[min(max(align * int(round(_log(r, low, high) / align)), low), case["size"]) for _a in range(3)]
            for _ in range(case["count"])]


def _queries(case, seed, fields, low, high, align):
    """(field, (lo, hi), relative tolerance) of sub-boxes, seeded places and tolerances."""
    r = random.Random(int(seed) + 977)
    out = []
    for sides in _sides(case, low, high, align):
        lo, hi = [], []
        for s in sides:
            o = align * r.randint(0, (case["size"] - s) // align)
            lo.append(o)
            hi.append(o + s)
        out.append((r.randrange(fields), (lo, hi), 10.0 ** r.uniform(-0.9 * case["n"], -1.0)))
    return out


def _side_by_side(boxes, dt, dtype=None):
    """One buffer for all boxes' results, each on a 256-byte boundary, and its parts."""
    sizes = [math.prod(h - l for l, h in zip(*b)) for b in boxes]
    step = 256 // _T[dt].itemsize
    at = np.concatenate([[0], np.cumsum([-(-v // step) * step for v in sizes])])
    buf = torch.zeros(int(at[-1]), dtype=dtype or _T[dt], device="cuda")
    return buf, [buf[int(at[j]):int(at[j]) + v] for j, v in enumerate(sizes)]


# ---- a program's state, and one pass of it ------------------------------------------


def prepare(case, seed):
    kind, dt = case["kind"], case["dtype"]
    s = dict(case)
    if kind in ("compress", "roundtrip"):
        s["x"] = _field(case["field"], _shape_of(case), dt, seed)
        if kind == "compress":
            s["archive"] = _archive_for(case)
    elif kind in ("retrieve", "sweep", "checkpoint"):
        x = _field(case["field"], _shape_of(case), dt, seed)
        s["tau"] = _schedule(x, case)
        s["st"] = pcz.compress(x, s["tau"])
        if kind != "checkpoint":
            s["out"] = torch.empty_like(x)
        else:
            s["archive"] = _archive_for(case)
            s["file"] = np.zeros(3 * x.numel() * x.element_size() + (1 << 20), dtype=np.uint8)
    elif kind in ("box", "boxes", "serve"):
        nf = case.get("fields", 1)
        s["sts"], s["taus"], ranges = [], [], []
        for f in range(nf):
            x = _field("powerlaw", [case["size"]] * 3, dt, seed * 64 + f)
            tau = pcz.field_tau_schedule(x, "decade", case["n"], param=1 if case["n"] > 8 else 2)
            lo, hi = pcz.field_range(x)
            ranges.append(hi - lo)
            s["taus"].append(tau)
            s["sts"].append(pcz.compress(x, tau))
        if kind == "box":
            r = random.Random(int(seed))
            lo = [r.randint(0, case["size"] - case["side"]) for _ in range(3)]
            s["box"] = (lo, [v + case["side"] for v in lo])
            s["tau"] = s["taus"][0][case["k"] - 1]
        elif kind == "boxes":
            qs = _queries(case, seed, nf, case["low"], case["high"], 1)
            s["streams"] = [s["sts"][f] for f, _b, _t in qs]
            s["boxes"] = [b for _f, b, _t in qs]
            s["ks"] = [s["sts"][f].query_k(max(t * ranges[f], s["taus"][f][-1])) for f, _b, t in qs]
            s["outs"] = [torch.empty([h - l for l, h in zip(*b)], dtype=_T[dt], device="cuda") for b in s["boxes"]]
        else:
            qs = _queries(case, seed, nf, 8, case["size"], 4)
            s["server"] = pcz.Server(20 * 10 ** 9, max_batch=512)
            for st in s["sts"]:
                s["server"].add_field(st)
            s["queries"] = [(f, b, max(t * ranges[f], s["taus"][f][-1]), 0) for f, b, t in qs]
            s["arrivals"] = [0.0] * len(qs)
            s["buffer"], s["outs"] = _side_by_side([b for _f, b, _t in qs], dt)
            s["server"].replay(s["queries"], s["arrivals"], s["outs"])  # a server that is up
    elif kind == "batch":
        s["shapes"] = _batch_shapes(case["count"], case["shapes"])
        s["xs"] = [_field("gaussians" if (j // 2) % 2 == 0 else "powerlaw", sh, dt, seed * 64 + j)
                   for j, sh in enumerate(s["shapes"])]
        s["taus"] = [pcz.field_tau_schedule(x, "decade", case["n"]) for x in s["xs"]]
        s["plan"] = pcz.Batch(s["shapes"], _T[dt], case["n"])
        s["plan"].compress(s["xs"], s["taus"])  # the plan picks its schedule on its first step
        s["outs"] = [torch.empty_like(x) for x in s["xs"]]
    else:
        s["u"], s["v"], s["w"] = (4.0 * _field("powerlaw", _shape_of(case), dt, 3 * seed + j) for j in range(3))
        s["om"], s["wzz"] = torch.empty_like(s["u"]), torch.empty_like(s["u"])
    return s


class _Array:
    """Device memory of a Streams object as a tensor that keeps the object alive."""

    def __init__(self, owner, ptr, count, typestr):
        self.owner = owner
        self.__cuda_array_interface__ = dict(shape=(count,), typestr=typestr, data=(ptr, False), version=3, strides=None,
                                             stream=None)


def _archive_for(case):
    """A program's buffer for the payloads of one field."""
    values = math.prod(_shape_of(case))
    return torch.zeros(2 * values * _T[case["dtype"]].itemsize // 8 + 4096, dtype=torch.int64, device="cuda")


def _stored(st, archive):
    """The payloads moved into the program's buffer, back to back; the index
    where it lies on the device; sizes and tolerances as computed."""
    out = dict(payload=archive, words=[], chunk_word=[], brick_len=[], measured=[])
    at = 0
    for i in range(st.n):
        pl, cw, bl, nw, nc, nb = st.device_ptrs(i)
        archive[at:at + nw].copy_(torch.as_tensor(_Array(st, pl, nw, "<i8"), device="cuda"))
        at += nw
        out["words"].append(nw)
        out["chunk_word"].append(torch.as_tensor(_Array(st, cw, nc, "<i8"), device="cuda"))
        out["brick_len"].append(torch.as_tensor(_Array(st, bl, nb, "<i2"), device="cuda"))
        out["measured"].append(st.measured_error(i))
    out["words"] = np.array(out["words"], dtype=np.int64)
    out["measured"] = np.array(out["measured"], dtype=np.float64)
    return out


def _summary(st):
    """Bits and index bytes of every component, and its tolerances."""
    info = [st.info(i) for i in range(st.n)]
    return (np.array([v[1:] for v in info], dtype=np.int64),
            np.array([(v[0], st.measured_error(i)) for i, v in enumerate(info)], dtype=np.float64))


def run(s):
    kind = s["kind"]
    if kind == "compress":
        return _stored(pcz.compress(s["x"], _schedule(s["x"], s)), s["archive"])
    if kind == "roundtrip":
        st = pcz.compress(s["x"], _schedule(s["x"], s))
        ks = range(1, st.n + 1) if s["all_k"] else (st.n,)
        return dict(streams=_summary(st), fields=[st.retrieve(k=k) for k in ks])
    if kind == "retrieve":
        return s["st"].retrieve(tau=s["tau"][s["k"] - 1], out=s["out"])
    if kind == "sweep":
        s["st"].retrieve(k=1, out=s["out"])
        for k in range(2, s["k"] + 1):
            s["st"].refine(k - 1, k, s["out"])
        return s["out"]
    if kind == "box":
        return s["sts"][0].retrieve(tau=s["tau"], box=s["box"])
    if kind == "boxes":
        return _joined(pcz.retrieve_batch(s["streams"], s["ks"], s["boxes"], s["outs"]))
    if kind == "serve":
        s["server"].replay(s["queries"], s["arrivals"], s["outs"])
        return s["buffer"]
    if kind == "batch":
        sts = s["plan"].compress(s["xs"], s["taus"])
        return pcz.retrieve_batch(sts, [s["n"]] * len(sts), outs=s["outs"])
    if kind == "checkpoint":
        data = s["st"].serialize()
        s["file"][:len(data)] = np.frombuffer(data, dtype=np.uint8)
        return dict(data=s["file"], size=len(data), streams=_stored(pcz.Streams.deserialize(data), s["archive"]))
    pcz.fd_vorticity_z(s["u"], s["v"], s["h"], out=s["om"])
    pcz.fd_second(s["w"], 2, s["h"], out=s["wzz"])
    return s["om"], s["wzz"]


def _joined(outs):
    """At most 64 results: a list of more is handed on as lists of equal share."""
    if len(outs) <= 64:
        return outs
    per = -(-len(outs) // 64)
    return [torch.cat([t.reshape(-1) for t in outs[i:i + per]]) for i in range(0, len(outs), per)]


# ---- the least work ------------------------------------------------------------------


def _rate(case, k=None, field=None):
    """About the bits per value of k components, index included, as coded
    fields of these kinds have: the first component by the field's spectrum,
    each further decade of tolerance (or binary step of 2^-4) some 5 bits more,
    in 2D 6.5."""
    n = case["n"] if k is None else k
    first = {"powerlaw": 11.5, "gaussians": 1.0, "fronts": 9.5}[field or case.get("field", "powerlaw")]
    more = 6.5 if case.get("ndims", 3) < 3 else 5.5 if case.get("schedule") == "binary" else 4.9
    return first + more * (n - 1)


def work(case):
    kind, b = case["kind"], _T[case["dtype"]].itemsize
    if kind == "derivative":
        v = case["nz"] * case["ny"] * case["nx"]
        return {"bytes": 5 * v * b, "flops": 8 * v}
    if kind in ("box", "boxes"):
        if kind == "box":
            v, k = case["side"] ** 3, case["k"]
        else:
            v = sum(math.prod(e) for e in _sides(case, case["low"], case["high"], 1))
            k = (case["n"] + 1) // 2
        return {"bytes": v * (b + _rate(case, k) / 8), "flops": v * k}
    if kind == "serve":
        v, k = sum(math.prod(e) for e in _sides(case, 8, case["size"], 4)), (case["n"] + 1) // 2
        return {"bytes": v * (b + _rate(case, k) / 8), "flops": v * k}
    if kind == "batch":
        v = sum(math.prod(sh) for sh in _batch_shapes(case["count"], case["shapes"]))
        return {"bytes": v * (2 * b + 2 * _rate(case, field="powerlaw") / 8), "flops": v * 3 * case["n"]}
    v = case["nz"] * case["ny"] * case["nx"]
    if kind == "compress":  # the field and its range, the streams
        return {"bytes": v * (b + _rate(case) / 8), "flops": v * 2 * case["n"]}
    if kind == "roundtrip":
        ks = range(1, case["n"] + 1) if case["all_k"] else (case["n"],)
        back = sum(_rate(case, k) / 8 + b for k in ks)
        return {"bytes": v * (b + _rate(case) / 8 + back), "flops": v * (2 * case["n"] + sum(ks))}
    if kind == "checkpoint":  # streams to the host and back
        return {"bytes": v * 4 * _rate(case) / 8, "flops": 0}
    if kind == "sweep":  # each refinement reads and writes the field
        return {"bytes": v * (_rate(case, case["k"]) / 8 + (2 * case["k"] - 1) * b), "flops": v * case["k"]}
    return {"bytes": v * (_rate(case, case["k"]) / 8 + b), "flops": v * case["k"]}


# ---- what the reconstructions stand for ------------------------------------------------


def _vorticity(u, v, h):
    def d(f, a):
        f = f.movedim(a, 0)
        o = torch.empty_like(f)
        o[1:-1] = (f[2:] - f[:-2]) / (2 * h)
        o[0] = (4 * f[1] - 3 * f[0] - f[2]) / (2 * h)
        o[-1] = (3 * f[-1] - 4 * f[-2] + f[-3]) / (2 * h)
        return o.movedim(0, a)

    return d(v, 2) - d(u, 1)


def _second_z(w, h):
    o = torch.empty_like(w)
    o[1:-1] = (w[2:] - 2 * w[1:-1] + w[:-2]) / (h * h)
    o[0] = (2 * w[0] - 5 * w[1] + 4 * w[2] - w[3]) / (h * h)
    o[-1] = (2 * w[-1] - 5 * w[-2] + 4 * w[-3] - w[-4]) / (h * h)
    return o


def exact(case, seed):
    """The derivatives in 64 bits; for a reconstruction, the field that was
    coded (a reconstruction is as far from it as its tolerance allows).  The
    streams themselves are whole numbers and have no such value."""
    kind, dt = case["kind"], case["dtype"]
    if kind == "derivative":
        u, v, w = (4.0 * _field("powerlaw", _shape_of(case), dt, 3 * seed + j) for j in range(3))
        return _vorticity(u.double(), v.double(), case["h"]), _second_z(w.double(), case["h"])
    if kind in ("retrieve", "sweep"):
        return _field(case["field"], _shape_of(case), dt, seed).double()
    if kind == "roundtrip":
        x = _field(case["field"], _shape_of(case), dt, seed).double()
        return dict(streams=(None, None), fields=[x] * (case["n"] if case["all_k"] else 1))
    if kind == "box":
        x = _field("powerlaw", [case["size"]] * 3, dt, seed * 64)
        r = random.Random(int(seed))
        lo = [r.randint(0, case["size"] - case["side"]) for _ in range(3)]
        return x[tuple(slice(v, v + case["side"]) for v in lo)].double()
    if kind == "boxes":
        xs = [_field("powerlaw", [case["size"]] * 3, dt, seed * 64 + f) for f in range(case["fields"])]
        qs = _queries(case, seed, case["fields"], case["low"], case["high"], 1)
        return _joined([xs[f][tuple(slice(l, h) for l, h in zip(*b))].double().contiguous() for f, b, _t in qs])
    if kind == "serve":
        xs = [_field("powerlaw", [case["size"]] * 3, dt, seed * 64 + f) for f in range(case["fields"])]
        qs = _queries(case, seed, case["fields"], 8, case["size"], 4)
        buf, outs = _side_by_side([b for _f, b, _t in qs], dt, torch.float64)
        for o, (f, b, _t) in zip(outs, qs):
            o.copy_(xs[f][tuple(slice(l, h) for l, h in zip(*b))].reshape(-1))
        return buf
    if kind == "batch":
        return [_field("gaussians" if (j // 2) % 2 == 0 else "powerlaw", sh, dt, seed * 64 + j).double()
                for j, sh in enumerate(_batch_shapes(case["count"], case["shapes"]))]
    return None
