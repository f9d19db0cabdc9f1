"""The measured cases: what a user of this library has it do, through its public binding.

A user holds a density field on the GPU, opens one context and calls one of the
measurement functions on field after field; the results come back as float64
arrays.  A case names the call (`kind`), the grid, the bins, the orders, the
field's type, the precision of the combination and the flags.
"""
import math
import weakref

import numpy as np
import torch

from paper_2210_10206_gb300 import sbg

PREC = {"fp32": sbg.SBG_PREC_FP32, "bf16x3": sbg.SBG_PREC_BF16X3, "tf32x3": sbg.SBG_PREC_TF32X3}

# One context serves every field of one kind of measurement, as a program that
# works through a set of snapshots keeps it; it goes when the last state does.
_contexts = weakref.WeakValueDictionary()


def _case(name, kind, n, nbins, hi, **more):
    c = dict(name=name, kind=kind, n=n, nfields=1, nbins=nbins, lo=2.0, hi=float(hi), log=False, lmax3=-1, lmax4=-1,
             dtype="float32", prec="fp32", normalized=False, autotune=True, sigma=1.0, slope=-2.0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one small 2D map, 3PCF only; latency and launches
        _case("projected 64 3pcf", "projected", 64, 4, 14, lmax3=4, dtype="float64"),
        # the allocation-free entry point inside a caller's own stream
        _case("noalloc 128 3pcf", "noalloc", 128, 7, 16, lmax3=5),
        # a column-density map at ordinary size: 10 bins, mmax 5, both statistics
        _case("projected 256 3+4pcf", "projected", 256, 10, 32, lmax3=5, lmax4=5),
        # the largest map with the most bins
        _case("projected 1024 20 bins", "projected", 1024, 20, 128, lmax3=5, lmax4=5, log=True),
        # snapshots of uneven sizes (128^2 .. 1024^2) in one call, high order, tensor cores
        _case("batch 16 uneven bf16x3", "batch", 1024, 10, 128, nfields=16, lmax3=10, lmax4=10, log=True,
              prec="bf16x3", autotune=False, sigma=1.2, slope=-8.0 / 3.0),
        # an odd number of slices of a simulation cube, normalised
        _case("slices 37 of 256", "slices", 256, 5, 32, nfields=37, lmax3=5, lmax4=5, normalized=True),
        # a small test box, both statistics: launches and tails
        _case("full 32 3+4pcf", "full", 32, 5, 12, lmax3=2, lmax4=2, dtype="float64"),
        # the ordinary 3D measurement in plain FP32
        _case("full 128 3+4pcf", "full", 128, 8, 18, lmax3=5, lmax4=3, sigma=1.2, slope=-3.0),
        # the parity-odd 4PCF, at the accurate tensor-core precision
        _case("full odd 128 tf32x3", "odd", 128, 7, 16, lmax4=4, prec="tf32x3", autotune=False, sigma=1.2, slope=-3.0),
        # the benchmark field, tensor cores (autotune off: launch choices, and so the last bits, repeat)
        _case("full 256 4pcf bf16x3", "full", 256, 10, 32, lmax4=4, prec="bf16x3", autotune=False, sigma=1.5,
              slope=-11.0 / 3.0),
        # the same field in plain FP32
        _case("full 256 4pcf fp32", "full", 256, 10, 32, lmax4=4, sigma=1.5, slope=-11.0 / 3.0),
        # the largest grid, whose kernel spectra do not fit: streamed over (l, m)
        _case("full 512 3pcf bf16x3", "full", 512, 20, 62, lmax3=5, prec="bf16x3", autotune=False, sigma=1.5,
              slope=-11.0 / 3.0),
    ]


def draw(rng):
    kind = rng.choice(["projected", "projected", "full", "full", "batch", "slices", "noalloc", "odd", "large"])
    prec = rng.choice(["fp32", "fp32", "bf16x3", "tf32x3"])
    c = dict(kind=kind, nfields=1, lo=rng.choice([0.0, 1.0, 2.0]), log=False, lmax3=-1, lmax4=-1,
             dtype=rng.choice(["float32", "float32", "float64"]), prec=prec, normalized=rng.random() < 0.25,
             autotune=prec == "fp32", sigma=round(rng.uniform(0.5, 1.5), 3), slope=round(rng.uniform(-11.0 / 3.0, -2.0), 3))
    if kind in ("projected", "batch", "slices"):
        c["n"] = rng.choice([32, 64, 128, 256, 512, 1024]) if kind != "slices" else rng.choice([64, 128, 256])
        c["nbins"] = rng.randint(1, 20 if kind == "projected" else 11)
        m = rng.randint(0, 10)
        if kind == "projected" and c["nbins"] > 10:
            m = min(m, 5)
        which = rng.choice(["3", "4", "34", "34"])
        c["lmax3"], c["lmax4"] = (m if "3" in which else -1), (m if "4" in which else -1)
        c["nfields"] = {"projected": 1, "batch": rng.randint(2, 16), "slices": rng.randint(3, 41)}[kind]
        c["log"] = kind != "slices" and rng.random() < 0.4
    elif kind == "noalloc":
        c["n"], c["nbins"], c["lmax3"] = rng.choice([8, 16, 32, 64, 128, 256]), rng.randint(1, 10), rng.randint(0, 10)
        c["prec"], c["autotune"], c["normalized"] = "fp32", True, False
    elif kind == "large":
        c.update(kind="full", n=512, nbins=rng.randint(3, 18), lmax3=rng.randint(1, 5), dtype="float32")
    else:
        c["n"] = rng.choice([16, 32, 64, 128, 256])
        c["nbins"] = rng.randint(1, 9)
        if kind == "odd":
            c["lmax4"] = rng.randint(1, 4)
        else:
            which = rng.choice(["3", "4", "34", "34"])
            c["lmax3"] = rng.randint(0, 6) if "3" in which else -1
            c["lmax4"] = rng.randint(0, 4) if "4" in which else -1
    # the outermost edge: a large part of a small box, a sixth to a ninth of a large one
    n = c["n"]
    c["hi"] = round(n * (rng.uniform(0.3, 0.49) if n <= 32 else rng.uniform(0.11, 0.16)), 2)
    if c["log"]:
        c["lo"] = max(c["lo"], 1.0)
        c["normalized"] = False
    c["nbins"] = max(1, min(c["nbins"], int(_smallest(c) * c["hi"] / n - c["lo"])))
    return c


def _smallest(case):
    return max(32, case["n"] // 8) if case["kind"] == "batch" else case["n"]


def _sizes(case):
    """Sides of the batch's fields: n / 8 .. n, as many of each, in order of size."""
    sides = [s for s in (case["n"] // 8, case["n"] // 4, case["n"] // 2, case["n"]) if s >= 32]
    return sorted(sides[i % len(sides)] for i in range(case["nfields"]))


def _edges(case, n=None):
    hi = case["hi"] * (n or case["n"]) / case["n"]
    f = np.geomspace if case["log"] else np.linspace
    return f(case["lo"], hi, case["nbins"] + 1)


def _field(shape, seed, case):
    """A lognormal density contrast with a power-law spectrum, made on the GPU."""
    dt = torch.float64 if case["dtype"] == "float64" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda", dtype=dt))
    k2 = torch.zeros((1,) * len(shape), device="cuda", dtype=dt)
    for i, s in enumerate(shape):
        f = torch.fft.rfftfreq(s, device="cuda", dtype=dt) if i == len(shape) - 1 else torch.fft.fftfreq(s, device="cuda", dtype=dt)
        k2 = k2 + (f * f).reshape([-1 if j == i else 1 for j in range(len(shape))])
    k2.view(-1)[0] = 1.0
    amp = k2.pow_(case["slope"] / 4)
    amp.view(-1)[0] = 0.0
    x = torch.fft.irfftn(w.mul_(amp), s=shape)
    x = x * (case["sigma"] / x.std())
    return torch.exp(x - 0.5 * case["sigma"] ** 2) - 1.0


def _fields(case, seed):
    n = case["n"]
    if case["kind"] == "batch":
        return [_field((s, s), seed * 1000 + i, case) for i, s in enumerate(_sizes(case))]
    if case["kind"] == "slices":
        return torch.stack([_field((n, n), seed * 1000 + i, case) for i in range(case["nfields"])])
    return _field((n, n) if case["kind"] in ("projected", "noalloc") else (n, n, n), seed * 1000, case)


def prepare(case, seed):
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    ctx = _contexts.get(key)
    if ctx is None and case["kind"] != "noalloc":
        ctx = sbg.Context(0)
        if not case["autotune"]:
            sbg.sbg_set_autotune(ctx.h, 0)
        _contexts[key] = ctx
    state = dict(case=case, ctx=ctx, field=_fields(case, seed), out=None)
    nb, m = case["nbins"], max(case["lmax3"], case["lmax4"])
    if case["kind"] == "batch":
        state["edges"] = [_edges(case, s) for s in _sizes(case)]
    else:
        state["edges"] = _edges(case)
    # long results are written again in place, as a loop over snapshots does
    w, z3, z4 = 2 * m + 1, (m + 1, nb, nb, 2), (2 * m + 1, 2 * m + 1, nb, nb, nb, 2)
    if case["kind"] in ("batch", "slices"):
        state["out"] = (np.zeros((case["nfields"],) + z3) if case["lmax3"] >= 0 else None,
                        np.zeros((case["nfields"],) + z4) if case["lmax4"] >= 0 else None)
    elif case["kind"] == "noalloc":
        state["out"] = torch.zeros(z3, dtype=torch.float64, device="cuda")
    return state


def run(state):
    case, ctx, field, edges = state["case"], state["ctx"], state["field"], state["edges"]
    l3, l4, prec = case["lmax3"], case["lmax4"], PREC[case["prec"]]
    npcf = ((3,) if l3 >= 0 else ()) + ((4,) if l4 >= 0 else ())
    flags = sbg.SBG_SUBTRACT_MEAN | (sbg.SBG_NORMALIZED if case["normalized"] else 0)
    m = max(l3, l4)
    if case["kind"] == "noalloc":
        return sbg.sbg_projected3_noalloc(field, edges, m, flags, state["out"], torch.cuda.current_stream().cuda_stream)
    if case["kind"] == "projected":
        z = ctx.projected(field, edges, m, npcf, prec, flags)
    elif case["kind"] == "batch":
        z = state["out"]
        each = [(z[0][i] if l3 >= 0 else None, z[1][i] if l4 >= 0 else None) for i in range(case["nfields"])]
        ctx.projected_batch(field, edges, case["nbins"], m, npcf, prec, flags, each)
    elif case["kind"] == "slices":
        z = ctx.projected_slices(field, edges, m, npcf, prec, flags, state["out"])
    elif case["kind"] == "odd":
        z = ctx.full_odd(field, edges, l4, prec, flags)
    else:
        z = ctx.full(field, edges, l3 if l3 >= 0 else None, l4 if l4 >= 0 else None, prec, flags)
    if case["kind"] == "odd":
        return {"zeta4": z}
    return {"zeta3": z[0], "zeta4": z[1]}


# ---------------------------------------------------------------- the work --
def _lambdas(lmax, odd):
    return [(a, b, c) for a in range(lmax + 1) for b in range(lmax + 1) for c in range(abs(a - b), min(a + b, lmax) + 1)
            if (a + b + c) % 2 == (1 if odd else 0)]


def work(case):
    """Each field read and each result written once; the transforms of the binned
    coefficients and the delta-weighted products (m >= 0, b1 <= b2 <= b3)."""
    nb, l3, l4 = case["nbins"], case["lmax3"], case["lmax4"]
    m = max(l3, l4)
    esz = 8 if case["dtype"] == "float64" else 4
    three = case["kind"] in ("full", "odd")
    sides = _sizes(case) if case["kind"] == "batch" else [case["n"]] * (case["nfields"] if case["kind"] == "slices" else 1)
    pairs, triples = nb * (nb + 1) // 2, nb * (nb + 1) * (nb + 2) // 6
    bytes_, flops = 0.0, 0.0
    for n in sides:
        ng = float(n) ** (3 if three else 2)
        groups = (lambda x: (x + 1) * (x + 2) // 2) if three else (lambda x: x + 1)
        bytes_ += ng * esz
        flops += (1 + groups(m) * nb) * 5 * ng * math.log2(ng)
        if l3 >= 0:
            bytes_ += ((l3 + 1) * nb * nb if three else 2 * (l3 + 1) * nb * nb) * 8
            flops += groups(l3) * pairs * 8 * ng
        if l4 >= 0 and three:
            lam = _lambdas(l4, case["kind"] == "odd")
            terms = sum(1 for a, b, c in lam for i in range(-a, a + 1) for j in range(-b, b + 1) if 0 <= -(i + j) <= c)
            bytes_ += len(lam) * nb**3 * 8
            flops += terms * triples * 4 * ng
        elif l4 >= 0:
            w = 2 * l4 + 1
            bytes_ += w * w * nb**3 * 16
            flops += (3 * l4 * (l4 + 1) + 1) / 2 * triples * 8 * ng
    return {"bytes": bytes_, "flops": flops}


# --------------------------------------------------------------- 64 bits ----
def _bin_index(dim, n, edges):
    """|r|^2 and offsets of the minimum-image grid, and the 0/1 mask of each bin."""
    i = torch.arange(n, device="cuda")
    i = torch.where(i < n - i, i, i - n).double()
    ax = [i.reshape([-1 if j == k else 1 for j in range(dim)]) for k in range(dim)]
    r2 = sum(a * a for a in ax)
    e2 = [float(e) ** 2 for e in edges]
    e2 = [round(v) if abs(v - round(v)) <= 1e-9 * max(v, 1.0) else v for v in e2]
    masks = [(r2 > e2[b]) & (r2 <= e2[b + 1]) for b in range(len(e2) - 1)]
    return ax, r2, masks


def _coefficients(delta, edges, orders):
    """a(x) = sum_r K(r) delta(x + r) for every order and bin: {order: [bins, points]}."""
    dim, n = delta.dim(), delta.shape[0]
    ax, r2, masks = _bin_index(dim, n, edges)
    axes = tuple(range(dim))
    dh = torch.fft.fftn(delta, dim=axes)
    r = torch.sqrt(torch.where(r2 > 0, r2, torch.ones_like(r2)))
    y, x = ax[-2], ax[-1]
    got = {}
    for o in orders:
        if dim == 2:
            k = torch.conj(torch.complex(x / r, y / r) ** o)
        else:
            l, m = o
            t = ax[0] / r
            p0, p1 = torch.zeros_like(t), torch.full_like(t, (-1.0) ** m * math.prod(range(1, 2 * m, 2)))
            for j in range(m + 1, l + 1):
                p0, p1 = p1, ((2 * j - 1) * t * p1 - (j + m - 1) * p0) / (j - m)
            norm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m))
            k = torch.conj(torch.complex(x / r, y / r).expand(r.shape) ** m) * (norm * p1)
        got[o] = torch.stack([torch.fft.ifftn(dh * torch.fft.ifftn(torch.where(b, k, torch.zeros_like(k)), dim=axes), dim=axes).reshape(-1)
                              * float(delta.numel()) for b in masks])
    return got


def _three_j(a, b, c, i, j, k):
    """Wigner 3j symbol by Racah's sum."""
    f = math.factorial
    if i + j + k or c < abs(a - b) or c > a + b or abs(i) > a or abs(j) > b or abs(k) > c:
        return 0.0
    s = sum((-1) ** t / (f(t) * f(c - b + t + i) * f(c - a + t - j) * f(a + b - c - t) * f(a - t - i) * f(b - t + j))
            for t in range(max(0, b - c - i, a - c + j), min(a + b - c, a - i, b + j) + 1))
    tri = f(a + b - c) * f(a - b + c) * f(b + c - a) / f(a + b + c + 1)
    return (-1) ** (a - b - k) * math.sqrt(tri * f(a + i) * f(a - i) * f(b + j) * f(b - j) * f(c + k) * f(c - k)) * s


def _pair_sums(delta, a, second, third):
    """sum_x delta a[b1] second[b2] third[c] over blocks of points: [bins, bins, columns]."""
    out = 0
    for x0 in range(0, delta.numel(), 1 << 18):
        s = slice(x0, x0 + (1 << 18))
        p = ((delta[s] * a[:, s])[:, None, :] * second[None, :, s]).reshape(-1, delta[s].numel())
        out = out + p @ third[:, s].T
    return out.reshape(a.shape[0], second.shape[0], -1)


def _exact_projected(field, edges, case):
    l3, l4, nb, n = case["lmax3"], case["lmax4"], case["nbins"], field.shape[0]
    d = field.double()
    d = d - d.mean()
    m = max(l3, l4)
    c = _coefficients(d, edges, range(m + 1))
    dl = d.reshape(-1)
    z3 = z4 = None
    if l3 >= 0:
        z3 = torch.view_as_real(torch.stack([(dl * c[k]) @ torch.conj(c[k]).T for k in range(m + 1)]).resolve_conj())
    if l4 >= 0:
        z4 = torch.zeros((2 * m + 1, 2 * m + 1, nb, nb, nb), dtype=torch.complex128, device="cuda")
        at = lambda k: c[k] if k >= 0 else torch.conj(c[-k]).resolve_conj()  # noqa: E731
        for m1 in range(-m, m + 1):
            for m2 in range(m1, m + 1):
                if abs(m1 + m2) > m or m1 + m2 < 0:
                    continue
                v = _pair_sums(dl, at(m1), at(m2), at(-(m1 + m2)))
                for s, u in ((1, v), (-1, torch.conj(v).resolve_conj())):
                    z4[s * m1 + m, s * m2 + m] = u
                    z4[s * m2 + m, s * m1 + m] = u.transpose(0, 1)
        z4 = torch.view_as_real(z4)
    if case["normalized"]:
        _, _, masks = _bin_index(2, n, edges)
        vb = torch.stack([b.sum() for b in masks]).double()
        ng = float(n) ** 2
        ngal = float((d + 1).sum())
        nv = ngal / ng * vb
        if z3 is not None:
            z3 = z3 / (ngal * nv[:, None] * nv[None, :])[..., None]
        if z4 is not None:
            z4 = z4 / (ngal * nv[:, None, None] * nv[None, :, None] * nv[None, None, :])[..., None]
    return z3, z4


def _exact_full(field, edges, case):
    l3, l4, nb, n = case["lmax3"], case["lmax4"], case["nbins"], field.shape[0]
    d = field.double()
    d = d - d.mean()
    dl = d.reshape(-1)
    ls = max(l3, l4)
    c = _coefficients(d, edges, [(l, m) for l in range(ls + 1) for m in range(l + 1)])
    z3 = z4 = None
    if l3 >= 0:
        z3 = torch.stack([(-1) ** l / math.sqrt(2 * l + 1) * sum((1 if m == 0 else 2) * ((dl * c[l, m]) @ torch.conj(c[l, m]).T).real
                                                                 for m in range(l + 1)) for l in range(l3 + 1)])
    if l4 >= 0:
        odd = case["kind"] == "odd"
        lam = _lambdas(l4, odd)
        place = {t: i for i, t in enumerate(lam)}
        z4 = torch.zeros((len(lam), nb, nb, nb), dtype=torch.float64, device="cuda")
        at = lambda l, m: c[l, m] if m >= 0 else (-1) ** m * torch.conj(c[l, -m]).resolve_conj()  # noqa: E731
        for a in range(l4 + 1):
            for b in range(a, l4 + 1):
                for i in range(-a, a + 1):
                    for j in range(-b, b + 1):
                        # M and -M give conjugates (times the parity): one of the two is computed
                        if abs(i + j) > l4 or (i, j) < (0, 0) or (a == b and (i, j) < (j, i) and (j, i) >= (0, 0)):
                            continue
                        m3 = -(i + j)
                        legs = [l for l in range(max(abs(m3), abs(a - b)), min(l4, a + b) + 1) if (a, b, l) in place]
                        if not legs:
                            continue
                        v = _pair_sums(dl, at(a, i), at(b, j), torch.cat([at(l, m3) for l in legs]))
                        v = (v.imag if odd else v.real).reshape(nb, nb, len(legs), nb)
                        # terms this product serves: (M, and -M unless M = 0), and for a == b also M with i, j
                        # exchanged (the transposed bins); for a != b also the Lambda with a and b exchanged
                        mult = 1.0 if (i, j) == (0, 0) else 2.0
                        for k, l in enumerate(legs):
                            sgn = -1.0 if odd else 1.0
                            w = mult * sgn * (-1) ** (a + b + l) * _three_j(a, b, l, i, j, m3)
                            t = w * v[:, :, k]
                            z4[place[a, b, l]] += t
                            # exchanged order: 3j(b, a, l; j, i, m3) = (-1)^(a + b + l) 3j(a, b, l; i, j, m3)
                            u = (-1) ** (a + b + l) * t.transpose(0, 1)
                            if a != b:
                                z4[place[b, a, l]] += u
                            elif i != j and (j, i) >= (0, 0):
                                z4[place[a, b, l]] += u
    if case["normalized"]:
        _, _, masks = _bin_index(3, n, edges)
        vb = torch.stack([b.sum() for b in masks]).double()
        ngal = float((d + 1).sum())
        nv = ngal / float(n) ** 3 * vb
        if z3 is not None:
            z3 = z3 / (ngal * nv[:, None] * nv[None, :])
        if z4 is not None:
            z4 = z4 / (ngal * nv[:, None, None] * nv[None, :, None] * nv[None, None, :])
    return z3, z4


def exact(case, seed):
    w = work(case)
    if case["n"] >= 512 and case["kind"] == "full" or w["flops"] > 2.5e12:
        return None  # over 20 seconds of 64-bit work
    field = _fields(case, seed)
    if case["kind"] == "batch":
        z = [_exact_projected(f, _edges(case, f.shape[0]), case) for f in field]
    elif case["kind"] == "slices":
        z = [_exact_projected(f, _edges(case), case) for f in field]
    elif case["kind"] in ("projected", "noalloc"):
        z = _exact_projected(field, _edges(case), case)
        return z[0] if case["kind"] == "noalloc" else {"zeta3": z[0], "zeta4": z[1]}
    else:
        z = _exact_full(field, _edges(case), case)
        return {"zeta4": z[1]} if case["kind"] == "odd" else {"zeta3": z[0], "zeta4": z[1]}
    join = lambda k: torch.stack([t[k] for t in z]) if z[0][k] is not None else None  # noqa: E731
    return {"zeta3": join(0), "zeta4": join(1)}
