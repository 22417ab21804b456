"""What the speed of the library is measured on: calls of its public API that a
fit makes, over the sizes they come in.

A case is a plain dict:

  call    the entry point (see KINDS)
  dtype   "float32" or "float64"
  nxy, M  image side and number of uv points (cube, walkers: the largest side
          and the number of points of one observation; n: requests per batch)
  reach   largest baseline in units of 1/dxy, the uv radius over the sampling
          frequency of the image (0.5 would be its Nyquist frequency).  0.45
          is the small and the profile configuration's coverage; 0.2 is what
          get_image_size's defaults give (f_max = 2.5); 0.0146 is an ALMA
          array of 3 km at 100 GHz on pixels of 0.002"
  layout  "random": uniform angle, log-uniform radius; "tracks": Earth-rotation
          tracks of 43 antennas, 60 time steps, as many channels as M needs
  fwhm    primary-beam width in image widths (0: none); K: copies of the model
"""
import math

import numpy as np
import torch

import paper_1709_06999_gb300 as gal
from paper_1709_06999_gb300.api import Request, default_context

ARCSEC = math.pi / (180.0 * 3600.0)
DEV = "cuda"
SIDES_CUBE = (512, 1024, 2048)
KINDS = ("chi2_image", "chi2_profile", "sample_image", "sample_profile", "chi2_arrays",
         "chi2_multi", "cube", "walkers")


def _case(name, call, dtype, nxy, M, reach, layout, **more):
    return dict(name=name, call=call, dtype=dtype, nxy=nxy, M=M, reach=reach, layout=layout,
                fwhm=more.get("fwhm", 0.0), K=more.get("K", 1), n=more.get("n", 1))


def listed():
    return [
        # a small map of a short observation: the time of a call is its launches
        _case("image_f64_256", "chi2_image", "float64", 256, 10_000, 0.45, "random"),
        # the paper's own calling convention: every call brings the data arrays
        _case("arrays_f64_512", "chi2_arrays", "float64", 512, 100_003, 0.2, "tracks"),
        # model visibilities of a disc, to plot or to subtract; an odd length
        _case("sample_profile_f32_512", "sample_profile", "float32", 512, 123_457, 0.2, "tracks"),
        # one likelihood of an axisymmetric disc fit, in both precisions
        _case("profile_f32_1024", "chi2_profile", "float32", 1024, 1_000_000, 0.45, "random"),
        _case("profile_f64_1024", "chi2_profile", "float64", 1024, 1_000_000, 0.45, "random"),
        # model visibilities of an image in the precision most fits run in
        _case("sample_image_f64_2048", "sample_image", "float64", 2048, 777_777, 0.2, "tracks"),
        # one likelihood of a large image over an ALMA data set, in both precisions
        _case("image_f32_4096", "chi2_image", "float32", 4096, 5_000_000, 0.0146, "tracks"),
        _case("image_f64_4096", "chi2_image", "float64", 4096, 5_000_000, 0.0146, "tracks"),
        # the channels of a spectral cube in one batch: images of three sizes,
        # every channel with its own points
        _case("cube_f32_64", "cube", "float32", 2048, 1_000_000, 0.0146, "tracks", n=64),
        # an ensemble step of a sampler: 64 discs against one observation
        _case("walkers_f32_64", "walkers", "float32", 1024, 1_000_000, 0.45, "random", n=64),
        # four displaced copies of one model (a multiple system)
        _case("multi_f32_2048", "chi2_multi", "float32", 2048, 2_000_003, 0.2, "tracks", K=4),
        # the largest image, seen through the primary beam, long baselines
        _case("beam_f32_8192", "chi2_image", "float32", 8192, 5_000_000, 0.2, "tracks", fwhm=0.6),
    ]


def draw(rng):
    call = rng.choice(KINDS)
    dtype = rng.choice(("float32", "float64")) if call not in ("cube", "walkers") else "float32"
    reach = round(math.exp(rng.uniform(math.log(0.0146), math.log(0.45))), 5)
    layout = rng.choice(("random", "tracks"))
    lg = rng.uniform(math.log(10_000), math.log(5_000_000))
    c = _case("", call, dtype, 0, int(math.exp(lg)), reach, layout)
    del c["name"]
    if call == "cube":
        # 0.11 of the 2048-pixel channels' frequency is 0.44 of the 512-pixel ones'
        c.update(nxy=2048, M=int(math.exp(rng.uniform(math.log(1e5), math.log(1e6)))),
                 n=rng.randint(8, 64), reach=min(reach, 0.11))
    elif call == "walkers":
        c.update(nxy=rng.choice((256, 512, 1024)), n=rng.randint(4, 64), M=min(c["M"], 1_000_000))
    elif call == "chi2_arrays":
        c.update(nxy=rng.choice((256, 512, 1024, 2048)), M=min(c["M"], 2_000_000))
    elif call.endswith("profile"):
        c.update(nxy=rng.choice((128, 256, 512, 1024, 2048)))
    else:
        c.update(nxy=rng.choice((64, 128, 256, 512, 1024, 2048, 4096)
                                + ((8192,) if dtype == "float32" else ())))
    if call == "chi2_multi":
        c.update(K=rng.randint(2, 8))
    if call == "chi2_image" and rng.random() < 0.25:
        c.update(fwhm=0.6)
    return c


# ---------------------------------------------------------------------------
# inputs, made on the device from the seed alone
# ---------------------------------------------------------------------------
def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)


def _uv(g, M, rho_max, layout):
    if layout == "random":
        ang = _uniform(g, M, 0.0, 2.0 * math.pi)
        rad = torch.exp(_uniform(g, M, math.log(rho_max / 450.0), math.log(rho_max)))
        return rad * torch.cos(ang), rad * torch.sin(ang)
    lat, dec, n_ant, n_time = math.radians(-23.0), math.radians(-35.0), 43, 60
    rad = torch.exp(_uniform(g, n_ant, math.log(15.0), math.log(3000.0)))
    az = _uniform(g, n_ant, 0.0, 2.0 * math.pi)
    i, j = torch.triu_indices(n_ant, n_ant, 1, device=DEV)
    be = (rad * torch.sin(az))[j] - (rad * torch.sin(az))[i]
    bn = (rad * torch.cos(az))[j] - (rad * torch.cos(az))[i]
    H = torch.linspace(-2.0, 2.0, n_time, device=DEV, dtype=torch.float64)[:, None] * (math.pi / 12)
    X, Z = -math.sin(lat) * bn, math.cos(lat) * bn
    u = (torch.sin(H) * X + torch.cos(H) * be).reshape(-1)
    v = (-math.sin(dec) * torch.cos(H) * X + math.sin(dec) * torch.sin(H) * be
         + math.cos(dec) * Z).reshape(-1)
    chans = max(1, -(-M // u.numel()))
    f = torch.linspace(96.25, 103.75, chans, device=DEV, dtype=torch.float64)[:, None]
    u, v = (f * u).reshape(-1)[:M], (f * v).reshape(-1)[:M]
    s = rho_max / torch.sqrt(u * u + v * v).max()
    return u * s, v * s


def _observation(g, M, rho_max, layout, dtype):
    """u, v, Re, Im, w: a 1 Jy Gaussian source of the models' size plus noise."""
    u, v = _uv(g, M, rho_max, layout)
    w = _uniform(g, M, 0.5, 2.0)
    sig = 1.0 / torch.sqrt(w)
    n = torch.randn(2, M, generator=g, device=DEV, dtype=torch.float64)
    V = torch.exp(-2.0 * math.pi ** 2 * (0.2 * ARCSEC) ** 2 * (u * u + v * v))
    return [t.to(dtype).contiguous() for t in (u, v, V + n[0] * sig, n[1] * sig, w)]


def _image(g, nxy, dxy, dtype):
    """Three elliptical Gaussians and an exponential disc, a few tenths of the field."""
    fov = nxy * dxy
    x = (nxy // 2 - torch.arange(nxy, device=DEV, dtype=torch.float64)) * dxy
    X, Y = x[None, :], x[:, None]
    img = torch.exp(-torch.sqrt(X * X + Y * Y) / (0.03 * fov))
    img = img / img.sum()
    for p in _uniform(g, (3, 6), 0.0, 1.0).tolist():
        s1, s2 = sorted(((0.005 + 0.03 * p[0]) * fov, (0.005 + 0.03 * p[1]) * fov))
        x0, y0, pa = (p[2] - 0.5) * 0.25 * fov, (p[3] - 0.5) * 0.25 * fov, math.pi * p[4]
        a = (X - x0) * math.sin(pa) + (Y - y0) * math.cos(pa)
        b = (X - x0) * math.cos(pa) - (Y - y0) * math.sin(pa)
        img = img + (0.1 + 0.9 * p[5]) * dxy * dxy / (2 * math.pi * s1 * s2) * torch.exp(
            -0.5 * ((a / s2) ** 2 + (b / s1) ** 2))
    return img.to(dtype).contiguous()


def _profile(p, nxy, dxy, dtype):
    """A Gaussian ring times a power law, 8192 samples out to 0.88 of the field, as Jy/sr."""
    fov, nr = nxy * dxy, 8192
    dR = 0.88 * fov / nr
    r = dR / 2 + dR * torch.arange(nr, device=DEV, dtype=torch.float64)
    r0, width, power = (0.06 + 0.08 * p[0]) * fov, (0.01 + 0.02 * p[1]) * fov, -p[2]
    I = torch.exp(-(((r - r0) / width) ** 2)) * (r / (0.2 * fov)) ** power
    I = I / (2 * math.pi * r0 * width * math.sqrt(math.pi))  # of the order of 1 Jy in all
    return I.to(dtype).contiguous(), dR / 2, dR


def _geometry(p, fov, inc=True):
    g = dict(dRA=(p[0] - 0.5) * 0.04 * fov, dDec=(p[1] - 0.5) * 0.04 * fov, PA=math.pi * p[2])
    return dict(g, inc=math.radians(70.0 * p[3])) if inc else g


def _inputs(case, seed):
    """Everything of a case as a dict of tensors and numbers: what prepare() hands to the
    library and exact() evaluates."""
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    dtype, nxy, call = getattr(torch, case["dtype"]), case["nxy"], case["call"]
    fov = 8.192 * ARCSEC
    dxy = fov / nxy
    p = _uniform(g, (max(1, case["n"]), 8), 0.0, 1.0).tolist()
    if call == "cube":
        rs = np.random.default_rng(int(seed))
        reqs = []
        for k in range(case["n"]):
            n = int(rs.choice(SIDES_CUBE))
            m = int(rs.integers(case["M"] // 10, case["M"] + 1))
            # baselines do not depend on the side a channel is imaged at
            reqs.append(dict(obs=_observation(g, m, case["reach"] * 2048 / fov, case["layout"], dtype),
                             image=_image(g, n, fov / n, dtype), dxy=fov / n,
                             geo=_geometry(p[0], fov, False)))
        return dict(reqs=reqs)
    obs = _observation(g, case["M"], case["reach"] / dxy, case["layout"], dtype)
    if call == "walkers":
        reqs = []
        for k in range(case["n"]):
            I, Rmin, dR = _profile(p[k][4:], nxy, dxy, dtype)
            reqs.append(dict(obs=obs, I=I, Rmin=Rmin, dR=dR, nxy=nxy, dxy=dxy,
                             geo=_geometry(p[k], fov)))
        return dict(reqs=reqs)
    q = dict(obs=obs, dxy=dxy, nxy=nxy)
    if call.endswith("profile"):
        q["I"], q["Rmin"], q["dR"] = _profile(p[0][4:], nxy, dxy, dtype)
        q["geo"] = _geometry(p[0], fov)
    else:
        q["image"] = _image(g, nxy, dxy, dtype)
        q["geo"] = _geometry(p[0], fov, False)
    q["fwhm"] = case["fwhm"] * fov
    if call == "chi2_multi":
        o = _uniform(g, (3, case["K"]), 0.0, 1.0).tolist()
        q["sources"] = ([(x - 0.5) * 0.1 * fov for x in o[0]], [(x - 0.5) * 0.1 * fov for x in o[1]],
                        [0.2 + x for x in o[2]])
    return q


def prepare(case, seed):
    q, call = _inputs(case, seed), case["call"]
    ctx = default_context()
    s = dict(call=call, ctx=ctx, q=q)
    if call in ("cube", "walkers"):
        shared, reqs = None, []
        for r in q["reqs"]:
            if call == "cube":
                reqs.append(Request(ctx.register(*r["obs"]), image=r["image"], dxy=r["dxy"], **r["geo"]))
            else:  # data that many models are compared with: kept in uv-plane order
                shared = shared or ctx.register(*r["obs"], z_order=True)
                reqs.append(Request(shared, intensity=r["I"], Rmin=r["Rmin"], dR=r["dR"],
                                    nxy=r["nxy"], dxy=r["dxy"], **r["geo"]))
        s["reqs"] = reqs
    elif call.startswith("chi2") and call != "chi2_arrays":
        s["obs"] = ctx.register(*q["obs"])
    return s


def run(s):
    call, ctx, q = s["call"], s["ctx"], s["q"]
    if call in ("cube", "walkers"):
        return ctx.chi2_batch(s["reqs"])
    geo = q["geo"]
    if call == "chi2_image":
        return ctx.chi2_image(q["image"], q["dxy"], s["obs"], pb_fwhm=q["fwhm"], **geo)
    if call == "chi2_profile":
        return ctx.chi2_profile(q["I"], q["Rmin"], q["dR"], q["nxy"], q["dxy"], s["obs"], **geo)
    if call == "chi2_arrays":
        return gal.chi2_image(q["image"], q["dxy"], *q["obs"], **geo)
    if call == "chi2_multi":
        return ctx.chi2_image_multi(q["image"], q["dxy"], s["obs"], *q["sources"], PA=geo["PA"])
    u, v = q["obs"][:2]
    if call == "sample_image":
        return ctx.sample_image(q["image"], q["dxy"], u, v, **geo)
    return ctx.sample_profile(q["I"], q["Rmin"], q["dR"], q["nxy"], q["dxy"], u, v, **geo)


def _work(call, nxy, M, e, reach, K):
    profile = call.endswith("profile") or call == "walkers"
    kc = min(nxy // 2 + 1, int(reach * nxy) + 2)
    b = (8192 if profile else nxy * nxy) * e
    b += M * (4 * e if call.startswith("sample") else 5 * e)
    lg = math.log2(nxy)
    # real rows, the kept columns; the image of a profile is even in both axes: a quarter
    f = (2.5 * nxy * nxy * lg + 5.0 * kc * nxy * lg) * (0.25 if profile else 1.0)
    f += M * (30.0 + 10.0 * K)
    return b, f


def work(case):
    """The image or profile and the points once each, the result once; the real row
    transforms, the columns the points reach, and the sampling of the points."""
    e = 8 if case["dtype"] == "float64" else 4
    if case["call"] == "cube":
        b = f = 0.0
        for n in SIDES_CUBE:
            x = _work("cube", n, 0.55 * case["M"], e, min(0.5, case["reach"] * 2048 / n), 1)
            b, f = b + x[0] * case["n"] / 3, f + x[1] * case["n"] / 3
    elif case["call"] == "walkers":  # one observation for all of them
        x = _work("walkers", case["nxy"], case["M"], e, case["reach"], 1)
        b = 5 * e * case["M"] + case["n"] * 8192 * e
        f = case["n"] * x[1]
    else:
        b, f = _work(case["call"], case["nxy"], case["M"], e, case["reach"], case["K"])
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# the same in 64 bits, written from the definitions with torch alone
# ---------------------------------------------------------------------------
def _exact_image(q):
    if "image" in q:
        img = q["image"].double()
    else:
        n, dxy = q["nxy"], q["dxy"]
        I = q["I"].double()
        x = (n // 2 - torch.arange(n, device=DEV, dtype=torch.float64)) * dxy
        r = torch.sqrt((x / math.cos(q["geo"]["inc"]))[None, :] ** 2 + x[:, None] ** 2)
        t = (r - q["Rmin"]) / q["dR"]
        k = torch.clamp(t.floor(), 0, I.numel() - 2).long()
        img = I[k] + (t - k) * (I[k + 1] - I[k])
        img = torch.where((t >= 0) & (t <= I.numel() - 1), img, torch.zeros_like(img))
        img[n // 2, n // 2] = I[0] - q["Rmin"] / q["dR"] * (I[1] - I[0])
        img = img * dxy * dxy
    if q.get("fwhm"):
        n, dxy, geo = img.shape[0], q["dxy"], q["geo"]
        x = (n // 2 - torch.arange(n, device=DEV, dtype=torch.float64)) * dxy
        c, s = math.cos(geo["PA"]), math.sin(geo["PA"])
        sx = x[None, :] * c + x[:, None] * s + geo["dRA"]
        sy = -x[None, :] * s + x[:, None] * c + geo["dDec"]
        img = img * torch.exp(-4 * math.log(2.0) * (sx * sx + sy * sy) / q["fwhm"] ** 2)
    return img


def _exact_vis(q):
    img, geo, dxy = _exact_image(q), q["geo"], q["dxy"]
    n = img.shape[0]
    G = torch.fft.fftshift(torch.fft.rfft2(torch.fft.fftshift(img)), dim=0)
    u, v = q["obs"][0].double(), q["obs"][1].double()
    c, s = math.cos(geo["PA"]), math.sin(geo["PA"])
    ur, vr = u * c - v * s, u * s + v * c
    neg = ur < 0
    iu = torch.clamp(ur.abs() * (n * dxy), 0, n // 2)
    iv = torch.clamp(n / 2 + torch.where(neg, -vr, vr) * (n * dxy), 0, n - 1)
    c0 = torch.clamp(iu.floor(), max=n // 2 - 1).long()
    r0 = torch.clamp(iv.floor(), max=n - 2).long()
    fu, fv = iu - c0, iv - r0
    V = ((1 - fv) * ((1 - fu) * G[r0, c0] + fu * G[r0, c0 + 1])
         + fv * ((1 - fu) * G[r0 + 1, c0] + fu * G[r0 + 1, c0 + 1]))
    V = torch.where(neg, V.conj(), V)
    dRA, dDec, amp = q.get("sources") or ([geo["dRA"]], [geo["dDec"]], [1.0])
    F = torch.zeros_like(V)
    for a, d, k in zip(dRA, dDec, amp):
        ph = 2 * math.pi * (u * a + v * d)
        F += k * torch.complex(torch.cos(ph), torch.sin(ph))
    return V * F


def _exact_one(q, call):
    V = _exact_vis(q)
    if call.startswith("sample"):
        return torch.view_as_real(V)
    re, im, w = (t.double() for t in q["obs"][2:])
    return (w * ((re - V.real) ** 2 + (im - V.imag) ** 2)).sum()


def exact(case, seed):
    q = _inputs(case, seed)
    if "reqs" in q:
        return torch.stack([_exact_one(r, "chi2") for r in q["reqs"]])
    return _exact_one(q, case["call"])
