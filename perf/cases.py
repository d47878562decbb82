"""The work that users of this framework have it do, as measurable cases.

listed() names the cases, draw() gives more of the same ranges, prepare()
makes what a program has in hand before the call (volume, mask, plan, output
buffers), run() is one pass through the public entry points, work() counts
what a pass cannot do without, and exact() evaluates the same maps in 64 bits
with plain torch.

Volumes and VOIs follow the repository's synthetic workloads (synth.py),
drawn on the GPU: i.i.d. uniform cubes, CT-like tissue classes with noise, and
MR-like smooth positive intensities with a blob VOI.
"""
import math

import torch

import paper_2609_19190_gb300 as fm
from paper_2609_19190_gb300.serve import Server

DEV = "cuda"
FBN, FBW = "fbn", "fbw"
FAMILY_ROWS = (("firstorder", 0, 18), ("glcm", 18, 42), ("glrlm", 42, 58), ("glszm", 58, 74),
               ("gldm", 74, 88), ("ngtdm", 88, 93), ("extras", 93, 102))
#: feature selections in use: the 93 benchmark maps, first order with GLCM,
#: first order alone, the whole default set of 101, the 102 scalar features
FEATURES = {"bench": range(93), "fo_glcm": range(42), "fo": range(18), "all": range(101),
            "scalar": range(102)}


def _case(name, kind, image, nx, ny, nz, voi, disc, bins, radius, features="bench", agg=0,
          delta=1, count=1, lo=0):
    return {"name": name, "kind": kind, "image": image, "nx": nx, "ny": ny, "nz": nz, "voi": voi,
            "disc": disc, "bins": bins, "radius": radius, "features": features, "agg": agg,
            "delta": delta, "count": count, "lo": lo}


def listed():
    return [
        # the smallest study: one tiny cube, first order and GLCM maps, where
        # launches and the slowest item count
        _case("tiny_r1", "map", "uniform", 32, 32, 32, 4224, FBN, 16, 1, "fo_glcm"),
        # one MR lesion (the paper's 61 x 55 x 39 crop with 50,613 voxels), 3^3 windows
        _case("lesion_r1", "map", "mr", 61, 55, 39, 50613, FBN, 32, 1),
        # one CT VOI at the repository's middle configuration: 25 HU bins, 5^3 windows
        _case("ct_r2", "map", "ct", 128, 128, 64, 200336, FBW, 25, 2),
        # the largest single volume: 2.0 M voxels, 64 levels, 7^3 windows, 93 maps
        _case("ct_large_r3", "map", "ct", 256, 256, 128, 2014083, FBN, 64, 3),
        # a cohort in one launch: ragged VOIs of mixed radius and bin count
        _case("batch_mixed", "batch", "ct", 128, 128, 64, 200000, FBN, 64, 3, count=32, lo=4000),
        # a burst of requests to the continuous-batching server, planned on arrival
        _case("served_burst", "served", "ct", 128, 128, 64, 200000, FBN, 64, 3, count=12, lo=4000),
        # fine discretisation (128 levels): windows with more levels than the
        # shared-memory paths hold
        _case("fine_levels_r2", "map", "mr", 61, 55, 39, 20011, FBN, 128, 2),
        # IBSI merged aggregation at GLCM distance 2, all 101 default maps
        _case("merged_r2", "map", "mr", 61, 55, 39, 30011, FBN, 32, 2, "all", agg=1, delta=2),
        # wide neighbourhoods (11^3)
        _case("wide_r5", "map", "ct", 64, 64, 64, 3001, FBN, 32, 5),
        # scalar extraction: one value per feature for the whole VOI
        _case("scalar_ct", "scalar", "ct", 128, 128, 64, 200336, FBW, 25, 1, "scalar"),
        # end to end through host buffers: image in, maps out
        _case("host_r1", "host", "ct", 128, 128, 64, 100003, FBW, 25, 1),
        # a new patient: plan, map, dense maps, release, for one small VOI
        _case("fresh_voi_r2", "fresh", "ct", 61, 55, 39, 9001, FBN, 32, 2),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["map"] * 6 + ["batch", "served", "scalar", "host", "fresh"])
    image = rng.choice(["ct", "ct", "mr", "uniform"])
    radius = rng.choice([1, 1, 2, 2, 3, 3, 4, 5])
    agg = int(rng.random() < 0.15)
    delta = 2 if rng.random() < 0.1 else 1
    # the costlier the window, the fewer voxels (no drawn case costs more than
    # the largest listed one)
    top = {1: 1500000, 2: 1000000, 3: 600000, 4: 6000, 5: 3000}[radius]
    disc, bins = (FBW, 25) if image == "ct" and rng.random() < 0.5 else (FBN, rng.choice([16, 32, 64]))
    if image != "ct" and radius <= 3 and rng.random() < 0.25:
        disc, bins = FBN, 128
    # windows beyond 24 levels or merged matrices take the general paths
    if bins == 128 or agg or delta > 1 or (image != "ct" and bins > 24):
        top = min(top, 20000 if radius >= 3 else 60000)
    count = 1
    if kind in ("batch", "served"):
        image, count, agg, delta = "ct", rng.randint(4, 24), 0, 1
        radius, disc, bins, top = rng.choice([1, 2, 3]), FBN, 64, 60000
    if kind == "scalar":
        radius, top = 1, 1000000
    if kind == "fresh":
        top = min(top, 50000)
    voi = size(1000, top)
    # a box that holds the VOI at about a third of its voxels, odd extents among them
    edge = (3.2 * voi) ** (1.0 / 3.0)
    nx = max(12, int(edge * rng.uniform(1.0, 1.4)))
    ny = max(12, int(edge * rng.uniform(0.9, 1.2)))
    nz = max(12, int(3.2 * voi / (nx * ny)) + 1)
    features = "scalar" if kind == "scalar" else rng.choice(["bench", "bench", "all", "fo_glcm", "fo"])
    if kind in ("batch", "served"):
        features = "bench"
    c = _case("", kind, image, nx, ny, nz, voi, disc, bins, radius, features, agg, delta, count,
              1000 if count > 1 else 0)
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _smooth(gen, shape, sigma):
    """Unit-variance smooth field (Gaussian low-pass, periodic)."""
    spec = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV))
    freqs = [torch.fft.fftfreq(n, device=DEV) for n in shape[:-1]]
    freqs.append(torch.fft.rfftfreq(shape[-1], device=DEV))
    for axis, f in enumerate(freqs):
        view = [1, 1, 1]
        view[axis] = -1
        spec = spec * torch.exp(-2.0 * (math.pi * sigma * f) ** 2).view(view)
    x = torch.fft.irfftn(spec, s=shape)
    x = x - x.mean()
    return x / x.std()


def _image(case, gen):
    shape = (case["nz"], case["ny"], case["nx"])
    if case["image"] == "uniform":
        return torch.randint(0, 256, shape, generator=gen, device=DEV).to(torch.int16)
    if case["image"] == "mr":
        x = 400.0 + 120.0 * _smooth(gen, shape, 3.0) + 20.0 * torch.randn(shape, generator=gen,
                                                                         device=DEV)
        return x.round().clamp(0, 4095).to(torch.int16)
    label = torch.stack([_smooth(gen, shape, 6.0) for _ in range(4)]).argmax(0)
    x = torch.zeros(shape, device=DEV)
    for c, (mu, sd) in enumerate(((-900.0, 60.0), (-50.0, 30.0), (40.0, 20.0), (300.0, 40.0))):
        x = torch.where(label == c, mu + sd * _smooth(gen, shape, 6.0), x)
    x = x + 15.0 * torch.randn(shape, generator=gen, device=DEV)
    return x.round().clamp(-32768, 32767).to(torch.int16)


def _mask(case, voi, gen):
    """uint8 VOI of exactly `voi` voxels (or all): an ellipsoid shaped like the
    box, for MR-like volumes a ragged blob."""
    shape = (case["nz"], case["ny"], case["nx"])
    if case["image"] == "mr":
        score = _smooth(gen, shape, 5.0)
    else:
        axes = [(torch.arange(n, device=DEV, dtype=torch.float32) - (n - 1) / 2) / n for n in shape]
        score = -(axes[0].view(-1, 1, 1) ** 2 + axes[1].view(1, -1, 1) ** 2
                  + axes[2].view(1, 1, -1) ** 2)
    flat = score.reshape(-1)
    m = torch.zeros(flat.numel(), dtype=torch.uint8, device=DEV)
    m[torch.sort(flat, descending=True, stable=True).indices[:voi]] = 1
    return m.view(shape)


def _params(case, radius, disc, bins):
    p = dict(kernel_radius=radius, aggregation=case["agg"], glcm_distance=case["delta"])
    if case["features"] != "bench":
        p["features"] = list(FEATURES[case["features"]])
    if disc == FBN:
        p.update(disc_mode=fm.FR_FBN, bin_count=bins)
    else:
        p.update(disc_mode=fm.FR_FBW, bin_width=float(bins))
    return fm.fr_map_params_init(case["nx"], case["ny"], case["nz"], **p)


def _units(case, seed):
    """The VOIs of a case: (image, mask, radius, disc, bins) each, from the seed."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if case["count"] == 1:
        image = _image(case, gen)
        return [(image, _mask(case, case["voi"], gen), case["radius"], case["disc"], case["bins"])]
    units = []
    for k in range(case["count"]):
        # sizes log-spaced over [lo, voi], each radius and bin count in turn
        f = k / (case["count"] - 1)
        voi = int(round(case["lo"] * (case["voi"] / case["lo"]) ** f))
        radius = 1 + (k + case["radius"]) % 3
        bins = (16, 32, 64)[(k // 3) % 3]
        disc = FBN if case["kind"] == "batch" or k % 2 == 0 else FBW
        units.append((_image(case, gen), _mask(case, voi, gen), radius, disc,
                      bins if disc == FBN else 25))
    return units


def _rows(case):
    return len(FEATURES[case["features"]])


def prepare(case, seed):
    units = _units(case, seed)
    kind = case["kind"]
    st = {"case": case, "kind": kind, "images": [u[0] for u in units]}
    params = [_params(case, u[2], u[3], u[4]) for u in units]
    # masks come from a contour tool in host memory, except the server's
    masks = [u[1] if kind == "served" else u[1].cpu() for u in units]
    if kind == "map":
        st["plan"] = fm.fr_map_plan(params[0], masks[0])
        st["out"] = torch.empty(_rows(case), st["plan"].n_voi, device=DEV)
    elif kind == "host":
        st["plan"] = fm.fr_map_plan(params[0], masks[0])
        st["image"] = units[0][0].cpu().pin_memory()
        st["out"] = torch.empty(_rows(case), st["plan"].n_voi, pin_memory=True)
    elif kind == "batch":
        st["batch"] = fm.fr_batch_plan(params, masks)
        st["outs"] = [torch.empty(st["batch"].n_rows[i], st["batch"].n_voi[i], device=DEV)
                      for i in range(len(units))]
    elif kind == "scalar":
        st["plan"] = fm.fr_scalar_plan(params[0], masks[0])
    elif kind == "served":
        st["server"] = Server(max_radius=3, max_slots=64)
        st["params"], st["masks"] = params, masks
        st["outs"] = [torch.empty(_rows(case), int(m.sum()), device=DEV) for m in masks]
        torch.cuda.synchronize()  # the server works on its own stream
    else:
        st["params"], st["masks"] = params, masks
    return st


def _by_family(case, out):
    """The maps as a program takes them: by feature family (views)."""
    ids = list(FEATURES[case["features"]])
    return {name: out[lo:min(hi, len(ids))] for name, lo, hi in FAMILY_ROWS if lo < len(ids)}


def run(st):
    kind = st["kind"]
    if kind == "map":
        return _by_family(st["case"], fm.fr_map_run(st["plan"], st["images"][0], st["out"]))
    if kind == "host":
        return _by_family(st["case"], fm.fr_map_run_host(st["plan"], st["image"], st["out"]))
    if kind == "batch":
        return fm.fr_batch_run(st["batch"], st["images"], st["outs"])
    if kind == "scalar":
        return fm.fr_scalar_run(st["plan"], st["images"][0])
    if kind == "served":
        srv, left = st["server"], 0
        for p, m, im, out in zip(st["params"], st["masks"], st["images"], st["outs"]):
            srv.add(p, m, im, out)
            left += 1
        while left:
            busy = srv.step(65536)
            for rid, status in srv.poll(wait=busy == 0):
                if status != 0:
                    raise RuntimeError("request ended with status %d" % status)
                srv.release(rid)
                left -= 1
        return st["outs"]
    plan = fm.fr_map_plan(st["params"][0], st["masks"][0])
    dense = fm.fr_scatter_dense(plan, fm.fr_map_run(plan, st["images"][0]))
    fm.fr_map_destroy(plan)
    return _by_family(st["case"], dense)


def work(case):
    """Bytes: image and mask-index of the VOI read once, maps written once.
    Operations: the increments, neighbour visits and sort steps that the
    definitions ask for per window (the roofline's window operations), plus
    the terms of the feature sums over the non-empty matrix cells."""
    rows = _rows(case)
    if case["kind"] == "scalar":
        n = case["voi"]
        return {"bytes": n * 6.0 + 8.0 * rows, "flops": n * (13.0 * 4 + 52 + 16)}
    total_b = total_f = 0.0
    for k in range(case["count"]):
        n, r = case["voi"], case["radius"]
        if case["count"] > 1:
            n = case["lo"] * (case["voi"] / case["lo"]) ** (k / (case["count"] - 1))
            r = 1 + (k + case["radius"]) % 3
        s, d = 2 * r + 1, case["delta"]
        w = s ** 3
        pairs = sum((s - d * abs(a)) * (s - d * abs(b)) * (s - d * abs(c))
                    for a, b, c in _DIRS if max(d * abs(a), d * abs(b), d * abs(c)) < s)
        ops = w * math.log2(w)
        if rows > 18:
            ops += 2 * pairs
        if rows > 42:
            ops += (13 + 13 + 26 + 26) * w
        out = 4.0 * rows * n
        if case["kind"] == "fresh":  # dense maps of the whole volume besides
            out += 4.0 * rows * case["nx"] * case["ny"] * case["nz"]
        total_b += 6.0 * n + out
        total_f += n * ops
    return {"bytes": total_b, "flops": total_f}


# ---------------------------------------------------------------- the same in 64 bits
_DIRS = [(dz, dy, dx) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)
         if (dz, dy, dx) > (0, 0, 0)]
_NAN = float("nan")


def _levels(img, mask, disc, bins):
    """Gray levels of the VOI (0 outside) and their number."""
    x = img.to(torch.int64)
    v = x[mask != 0]
    lo, hi = int(v.min()), int(v.max())
    if disc == FBN:
        ng = bins
        g = torch.ones_like(x) if hi == lo else ((x - lo) * ng // (hi - lo) + 1).clamp(1, ng)
    else:
        ng = int(math.floor((float(hi) - float(lo)) / float(bins))) + 1
        g = torch.floor((x.double() - float(lo)) / float(bins)).to(torch.int64) + 1
    return torch.where(mask != 0, g, torch.zeros_like(g)), ng


def _shift(x, d, fill=0):
    """y(u) = x(u + d) over the last three axes, `fill` beyond them."""
    out = torch.full_like(x, fill)
    src, dst = [Ellipsis], [Ellipsis]
    for k, n in zip(d, x.shape[-3:]):
        if abs(k) >= n:
            return out
        src.append(slice(max(k, 0), n + min(k, 0)))
        dst.append(slice(max(-k, 0), n + min(-k, 0)))
    out[tuple(dst)] = x[tuple(src)]
    return out


def _div(a, b):
    return torch.where(b == 0, torch.full_like(a, _NAN), a / torch.where(b == 0, torch.ones_like(b), b))


def _plogp(p):
    return -torch.where(p > 0, p * torch.log2(p.clamp_min(1e-300)), torch.zeros_like(p))


def _firstorder(raw, valid, hist, excess=True):
    n = valid.sum(1)
    N = n.double()
    x = raw.double()
    vd = valid.double()
    srt = torch.sort(torch.where(valid, raw, torch.full_like(raw, 1 << 40)), 1).values

    def at(k):
        return srt.gather(1, k.view(-1, 1)).view(-1)

    num = {}
    for q in (10, 25, 50, 75, 90):
        h = (n - 1) * q
        k, rem = h // 100, h % 100
        a, b = at(k), at(torch.minimum(k + 1, n - 1))
        num[q] = 100 * a + rem * (b - a)  # 100 P_q, exact
    s1 = (raw * valid).sum(1)
    s2 = (raw * raw * valid).sum(1).double()
    mu = s1.double() / N
    c = (x - mu.view(-1, 1)) * vd
    m2, m3, m4 = (c ** 2).sum(1) / N, (c ** 3).sum(1) / N, (c ** 4).sum(1) / N
    flat = at(torch.zeros_like(n)) == at(n - 1)
    zero = torch.zeros_like(m2)
    m2 = torch.where(flat, zero, m2)
    lo, hi = at(torch.zeros_like(n)).double(), at(n - 1).double()
    sub = valid & (100 * raw >= num[10].view(-1, 1)) & (100 * raw <= num[90].view(-1, 1))
    sd = sub.double()
    rn = sd.sum(1)
    rmu = _div((x * sd).sum(1), rn)
    rmad = _div(((x - rmu.view(-1, 1)).abs() * sd).sum(1), rn)
    p = hist / N.view(-1, 1)
    pq = {q: v.double() / 100 for q, v in num.items()}
    f = [s2, s2, _plogp(p).sum(1), lo, pq[10], pq[90], hi, mu, pq[50], pq[75] - pq[25], hi - lo,
         c.abs().sum(1) / N, rmad, (s2 / N).sqrt(), _div(m3, m2 ** 1.5),
         _div(m4, m2 ** 2) - (3.0 if excess else 0.0), m2, (p * p).sum(1)]
    extra = [((x - pq[50].view(-1, 1)).abs() * vd).sum(1) / N, _div(m2.sqrt(), s1.double() / N),
             _div((num[75] - num[25]).double(), (num[75] + num[25]).double())]
    return f, extra, m2.sqrt()


def _second_eigenvalue(P, px):
    """Second-largest |eigenvalue| of D^-1/2 P D^-1/2: the spectral radius of
    the deflated matrix, by repeated squaring and one Rayleigh quotient."""
    u = px.sqrt()
    den = u.unsqueeze(-1) * u.unsqueeze(-2)
    A = torch.where(den > 0, P / torch.where(den > 0, den, torch.ones_like(den)),
                    torch.zeros_like(P)) - den
    B = A
    for _ in range(18):
        B = B @ B
        B = B / B.abs().amax((-1, -2), keepdim=True).clamp_min(1e-300)
    norms = (B * B).sum(-2)
    v = B.gather(-1, norms.argmax(-1)[..., None, None].expand(*B.shape[:-1], 1))
    Av = A @ v
    return ((Av * Av).sum((-1, -2)) / (v * v).sum((-1, -2)).clamp_min(1e-300)).sqrt()


def _glcm(lv, rank, m, ng, delta, merged):
    """Per direction (or merged) GLCM features [n, matrices, 24] and the two extras."""
    n, dev = lv.shape[0], lv.device
    mats = []
    for k, d in enumerate(_DIRS):
        dd = tuple(delta * c for c in d)
        ok = (lv > 0) & (_shift(lv, dd) > 0)
        which, *_ = torch.nonzero(ok, as_tuple=True)
        mats.append((which, lv[ok], _shift(lv, dd)[ok], rank[ok], _shift(rank, dd)[ok]))
    if merged:
        mats = [tuple(torch.cat([x[k] for x in mats]) for k in range(5))]
    feats, extras = [], []
    for which, i, j, ri, rj in mats:
        def per(v):
            return torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, which, v.double())

        def hist(key, size):
            return torch.bincount(which * size + key, minlength=n * size).view(n, size).double()

        T = 2 * per(torch.ones_like(i))
        some = T > 0
        t = torch.where(some, T, torch.ones_like(T))
        P = hist(ri * m + rj, m * m).view(n, m, m)
        P = (P + P.transpose(1, 2)) / t.view(-1, 1, 1)
        px = P.sum(2)
        mux = per(i + j) / t
        sq = per(i * i + j * j)
        var_num = T * sq - per(i + j) ** 2
        autoc = 2 * per(i * j) / t
        cov_num = 2 * T * per(i * j) - per(i + j) ** 2
        cl = (i + j).double() - 2 * mux[which]
        kd, ks = (i - j).abs(), i + j
        pd = 2 * hist(kd, ng) / t.view(-1, 1)
        ps = 2 * hist(ks, 2 * ng + 1) / t.view(-1, 1)
        k1 = torch.arange(ng, dtype=torch.float64, device=dev)
        da = (k1 * pd).sum(1)
        hx, hxy = _plogp(px).sum(1), _plogp(P).sum((1, 2))
        # mutual information as a sum of nonnegative terms
        q = px.unsqueeze(2) * px.unsqueeze(1)
        x = torch.where(q > 0, (P - q) / torch.where(q > 0, q, torch.ones_like(q)), torch.zeros_like(q))
        g = torch.where(x.abs() < 1e-3, x * x * (0.5 - x / 6 + x * x / 12 - x ** 3 / 20 + x ** 4 / 30),
                        torch.where(x > -1, (1 + x) * torch.log1p(x.clamp_min(-1 + 1e-16)) - x,
                                    torch.ones_like(x)))
        mi = (q * g).sum((1, 2)) / math.log(2.0)
        present = (px > 0).sum(1)
        mcc = torch.where(present >= 2, _second_eigenvalue(P, px), torch.full_like(T, _NAN))
        sa = 2 * per(ks) / t
        sv = 2 * per((ks.double() - sa[which]) ** 2) / t
        f = [autoc, mux, 2 * per(cl ** 4) / t, 2 * per(cl ** 3) / t, 2 * per(cl ** 2) / t,
             2 * per(kd * kd) / t, _div(cov_num, var_num), da, _plogp(pd).sum(1),
             ((k1 - da.view(-1, 1)) ** 2 * pd).sum(1), (P * P).sum((1, 2)), hxy, _div(-mi, hx),
             torch.sqrt((-torch.expm1(-2 * mi)).clamp_min(0)),
             (pd / (1 + k1 * k1)).sum(1), (pd / (1 + k1 * k1 / (ng * ng))).sum(1),
             (pd / (1 + k1)).sum(1), (pd / (1 + k1 / ng)).sum(1),
             (pd[:, 1:] / k1[1:] ** 2).sum(1), P.amax((1, 2)), sa, _plogp(ps).sum(1),
             var_num / (t * t), mcc]
        nan = torch.full_like(T, _NAN)
        feats.append(torch.stack([torch.where(some, v, nan) for v in f], 1))
        extras.append(torch.stack([torch.where(some, v, nan) for v in (sv, da)], 1))
    return torch.stack(feats, 1).nanmean(1), torch.stack(extras, 1).nanmean(1)


def _cells(which, n, i, j, count, nv):
    """The 16 run-length / zone features from cells (matrix, level i, length
    j, count), every matrix with at least one run."""
    c, i, j = count.double(), i.double(), j.double()

    def per(v):
        return torch.zeros(n, dtype=torch.float64, device=c.device).index_add_(0, which, v)

    def squares(key):
        size = int(key.max()) + 1
        h = torch.zeros(n * size, dtype=torch.float64, device=c.device)
        h.index_add_(0, which * size + key.long(), c)
        return (h * h).view(n, size).sum(1)

    N = per(c)
    mi, mj = per(c * i) / N, per(c * j) / N
    gl, sz = squares(i), squares(j)
    return torch.stack([
        per(c / j ** 2) / N, per(c * j ** 2) / N, gl / N, gl / N ** 2, sz / N, sz / N ** 2, N / nv,
        per(c * (i - mi[which]) ** 2) / N, per(c * (j - mj[which]) ** 2) / N,
        per(_plogp(c / N[which])), per(c / i ** 2) / N, per(c * i ** 2) / N,
        per(c / (i * j) ** 2) / N, per(c * i ** 2 / j ** 2) / N, per(c * j ** 2 / i ** 2) / N,
        per(c * (i * j) ** 2) / N], 1)


def _count_cells(which, i, j):
    """Distinct (matrix, level, length) triples and how often each occurs."""
    wide = int(j.max()) + 1 if j.numel() else 1
    key, count = torch.unique((which * 256 + i) * wide + j, return_counts=True)
    return key // (256 * wide), key // wide % 256, key % wide, count


def _glrlm(lv, nv, merged):
    n = lv.shape[0]
    rows = []
    for d in _DIRS:
        back = tuple(-c for c in d)
        same = (lv > 0) & (lv == _shift(lv, d))
        start = (lv > 0) & ~_shift(same, back, False)
        length = torch.ones_like(lv)
        chain = same
        while bool(chain.any()):
            length = length + chain
            chain = same & _shift(chain, d, False)
        which, *_ = torch.nonzero(start, as_tuple=True)
        rows.append((which, lv[start], length[start]))
    if merged:
        rows = [tuple(torch.cat([r[k] for r in rows]) for k in range(3))]
        nv = 13 * nv
    out = []
    for which, i, j in rows:
        w, a, b, c = _count_cells(which, i, j)
        out.append(_cells(w, n, a, b, c, nv))
    return torch.stack(out, 1).mean(1)


def _glszm(lv, nv):
    n, cells = lv.shape[0], lv[0].numel()
    lab = torch.arange(1, n * cells + 1, device=lv.device).view(lv.shape) * (lv > 0)
    while True:
        new = lab
        for d in _DIRS:
            for sgn in (1, -1):
                dd = tuple(sgn * c for c in d)
                new = torch.where((lv > 0) & (lv == _shift(lv, dd)), torch.maximum(new, _shift(new, dd)), new)
        # a label names a voxel of the same zone: follow it
        flat = new.view(-1)
        new = torch.where(new > 0, flat[(new - 1).clamp_min(0).view(-1)].view(new.shape), new)
        if torch.equal(new, lab):
            break
        lab = new
    root, size = torch.unique(lab[lab > 0], return_counts=True)
    which, level = (root - 1) // cells, lv.view(-1)[root - 1]
    return _cells(*_relabel(n, *_count_cells(which, level, size)), nv)


def _relabel(n, w, i, j, c):
    return w, n, i, j, c


def _gldm_ngtdm(lv, valid, nv, ng):
    n = lv.shape[0]
    eq, num, tot = torch.zeros_like(lv), torch.zeros_like(lv), torch.zeros_like(lv)
    for d in _DIRS:
        for sgn in (1, -1):
            nb = _shift(lv, tuple(sgn * c for c in d))
            eq += (nb == lv) & valid
            num += (nb > 0)
            tot += nb
    which, *_ = torch.nonzero(valid, as_tuple=True)
    w, i, j, c = _count_cells(which, lv[valid], eq[valid] + 1)
    full = _cells(w, n, i, j, c, nv)
    gldm = full[:, [0, 1, 2, 4, 5, 7, 8, 9, 10, 11, 12, 13, 14, 15]]
    p = c.double() / nv[w]
    energy = torch.zeros(n, dtype=torch.float64, device=lv.device).index_add_(0, w, p * p)
    extra = [full[:, 3], torch.ones_like(energy), energy]
    has = valid & (num > 0)
    which, *_ = torch.nonzero(has, as_tuple=True)
    level = lv[has]
    dlt = (level.double() - tot[has].double() / num[has].double()).abs()
    dlt = torch.where(level * num[has] == tot[has], torch.zeros_like(dlt), dlt)
    ni = torch.zeros(n * (ng + 1), dtype=torch.float64, device=lv.device)
    si = torch.zeros_like(ni)
    ni.index_add_(0, which * (ng + 1) + level, torch.ones_like(dlt))
    si.index_add_(0, which * (ng + 1) + level, dlt)
    ni, si = ni.view(n, -1), si.view(n, -1)
    N = ni.sum(1)
    one = N.clamp_min(1).view(-1, 1)
    p, g = ni / one, torch.arange(ng + 1, dtype=torch.float64, device=lv.device)
    ngp = (ni > 0).sum(1).double()
    sps, ss = (p * si).sum(1), si.sum(1)
    both = (ni > 0).unsqueeze(2) & (ni > 0).unsqueeze(1)
    dg = (g.view(-1, 1) - g.view(1, -1))
    con = (p.unsqueeze(2) * p.unsqueeze(1) * dg ** 2).sum((1, 2))
    con = torch.where(ngp > 1, con / (ngp * (ngp - 1)).clamp_min(1) * ss / one.view(-1), torch.zeros_like(con))
    ip = g * ni
    bden = ((ip.unsqueeze(2) - ip.unsqueeze(1)).abs() * both).sum((1, 2)) / one.view(-1)
    psum = p.unsqueeze(2) + p.unsqueeze(1)
    ps = p * si
    cpl = (torch.where(both, dg.abs() * (ps.unsqueeze(2) + ps.unsqueeze(1)) / psum.clamp_min(1e-300),
                       torch.zeros_like(psum))).sum((1, 2)) / one.view(-1)
    stg = (torch.where(both, psum * dg ** 2, torch.zeros_like(psum))).sum((1, 2))
    f = [_div(torch.ones_like(sps), sps), con, _div(sps, bden), cpl, _div(stg, ss)]
    nan = torch.full_like(N, _NAN)
    return gldm, extra, torch.stack([torch.where(N > 0, v, nan) for v in f], 1)


def _windows(lv, raw, ng, count, delta, merged):
    """Features [n, count] (ids 0 .. count - 1) of n windows lv, raw [n, z, y, x]."""
    n = lv.shape[0]
    valid = lv > 0
    nv = valid.view(n, -1).sum(1).double()
    flat = lv.view(n, -1)
    hist = torch.zeros(n, ng + 1, dtype=torch.float64, device=lv.device)
    hist.scatter_add_(1, flat, valid.view(n, -1).double())
    fo, fo_extra, std = _firstorder(raw.view(n, -1), valid.view(n, -1), hist)
    out = [torch.stack(fo, 1)]
    if count > 18:
        rank_of = (hist > 0).long().cumsum(1) - 1
        m = max(1, int((hist > 0).sum(1).max()))
        rank = rank_of.gather(1, flat).clamp_min(0).view(lv.shape)
        glcm, glcm_extra = _glcm(lv, rank, m, ng, delta, merged)
        out.append(glcm)
    if count > 42:
        out += [_glrlm(lv, nv, merged), _glszm(lv, nv)]
        gldm, gldm_extra, ngtdm = _gldm_ngtdm(lv, valid, nv, ng)
        out += [gldm, ngtdm]
    if count > 93:
        out += [torch.stack(fo_extra, 1), glcm_extra, torch.stack(gldm_extra, 1)]
    if count > 101:
        out.append(std.view(-1, 1))
    return torch.cat(out, 1)


def _exact_maps(case, unit):
    img, mask, r, disc, bins = unit
    lv, ng = _levels(img, mask, disc, bins)
    s = 2 * r + 1
    pad = [r] * 6
    lvp = torch.nn.functional.pad(lv, pad)
    rawp = torch.nn.functional.pad(img.long() * (mask != 0), pad)
    _, py, px = lvp.shape
    o = torch.arange(s, device=lv.device)
    off = ((o.view(-1, 1, 1) * py + o.view(1, -1, 1)) * px + o.view(1, 1, -1)).reshape(-1)
    z, y, x = torch.nonzero(mask, as_tuple=True)
    corner = (z * py + y) * px + x
    count = _rows(case)
    step = max(64, min(8192, int(2e8 / (s ** 3 * 8 + ng * ng * 8))))
    out = []
    for k in range(0, corner.numel(), step):
        at = corner[k:k + step].view(-1, 1) + off
        shape = (at.shape[0], s, s, s)
        out.append(_windows(lvp.view(-1)[at].view(shape), rawp.view(-1)[at].view(shape), ng, count,
                            case["delta"], case["agg"] == 1))
    return torch.cat(out).t().contiguous()


def _affordable(case, voi, radius, bins):
    """Whether the 64-bit evaluation of one VOI stays within a few seconds."""
    levels = bins if case["image"] != "ct" else 24
    cost = voi * ((2 * radius + 1) ** 3 * 13 * 40.0 + 13 * min(levels, (2 * radius + 1) ** 3) ** 2 * 60.0)
    return cost < 3e11


def exact(case, seed):
    units = _units(case, seed)
    kind = case["kind"]
    if kind == "scalar":
        img, mask, _, disc, bins = units[0]
        if case["voi"] > 300000:
            return None
        lv, ng = _levels(img, mask, disc, bins)
        return _windows(lv[None], (img.long() * (mask != 0))[None], ng, 102, case["delta"],
                        case["agg"] == 1)[0]
    if case["count"] > 1:  # the smaller VOIs of a batch
        return [_exact_maps(case, u) if int(u[1].sum()) <= 6000 else None for u in units]
    if not _affordable(case, case["voi"], case["radius"], case["bins"]):
        return None
    maps = _exact_maps(case, units[0])
    if kind == "fresh":
        mask = units[0][1]
        dense = torch.full((maps.shape[0],) + tuple(mask.shape), _NAN, dtype=torch.float64,
                           device=maps.device)
        dense[:, mask != 0] = maps
        maps = dense
    return _by_family(case, maps)
