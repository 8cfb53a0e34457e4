"""The calls this library is measured on, and what they compute.

Twelve listed cases and a generator of further ones (``draw``), all through
the Python binding of the C ABI: Gonzalez selection (GON), the covering
radius, two-round MRG, EIM and the batched form, on float32 and int32 points,
with the float32, bf16 and fp16 sweeps.  The sizes are those of the
repository's workloads (10k x 2 int32, 1M x 10, 10M x 16 in Zipf parts,
8M x 64, 4,096 instances of mixed sizes), of its 2-D sweeps over k and n, and
odd ones between them.

The point sets are the shapes of the paper's synthetic sets: ``unif`` (a
uniform box), ``gau`` (isotropic Gaussian clusters of equal size) and ``unb``
(the same with half, in the batch 90%, of the points in one cluster).

Every output is compared exactly: a selection is defined on the canonical
float32 squared distance (t = x_j - c_j rounded, acc = fma(t, t, acc) in
coordinate order) with ties to the lowest index, and a radius on the float64
distance in coordinate order, so two correct implementations return the same
bits.  The fp8 sweep is left out: on these sets its 3-bit mantissa leaves most
points to the exact recheck, and no program would choose it.
"""
import math
import random

import torch

import paper_1604_03228_gb300 as kc

DEV = "cuda"
EPS, PHI = 0.1, 6.0


def listed():
    return [
        # The smallest call a program makes: 10,000 integer grid points in the
        # plane, ten centers; launches and latency count.
        dict(name="gon_i32_10k_d2_k10", method="gon", dtype="i32", sweep="f32", shape="unif", n=10_000, d=2, k=10),
        # The paper's 2-D sets (Unif, 100k points) at its largest k: a hundred
        # dependent steps of a few microseconds each.
        dict(name="gon_f32_100k_d2_k100", method="gon", dtype="f32", sweep="f32", shape="unif", n=100_000, d=2, k=100),
        # GON on a set that fits on chip (25 clusters), the repository's
        # ordinary workload, and the radius of its centers below.
        dict(name="gon_f32_1m_d10_k100", method="gon", dtype="f32", sweep="f32", shape="gau", clusters=25, n=1_000_000,
             d=10, k=100),
        # An embedding of no convenient width and an odd point count, without
        # cluster structure.
        dict(name="gon_f32_777777_d37_k50", method="gon", dtype="f32", sweep="f32", shape="unif", n=777_777, d=37, k=50),
        # The headline workload: 8M points of 64 coordinates, 1024 centers,
        # streamed from device memory; in float32 and with the bf16 sweep.
        dict(name="gon_f32_8m_d64_k1024", method="gon", dtype="f32", sweep="f32", shape="gau", clusters=100,
             n=8_000_000, d=64, k=1024),
        dict(name="gon_bf16_8m_d64_k1024", method="gon", dtype="f32", sweep="bf16", shape="gau", clusters=100,
             n=8_000_000, d=64, k=1024),
        # The solution value of a given center set: on the CUDA cores, and the
        # largest block on the tensor cores.
        dict(name="radius_f32_1m_d10_k100", method="radius", dtype="f32", shape="gau", clusters=25, n=1_000_000, d=10,
             k=100),
        dict(name="radius_f32_8m_d64_k1024", method="radius", dtype="f32", shape="gau", clusters=100, n=8_000_000, d=64,
             k=1024),
        # MRG: 64 parts of Zipf(1.1) sizes, GON on each, GON on their union.
        dict(name="mrg_f32_10m_d16_k200", method="mrg", dtype="f32", sweep="f32", shape="unif", n=10_000_000, d=16,
             k=200, m=64, zipf=1.1),
        # EIM: the paper's own 2-D setting, and the large one whose distance
        # blocks run on the tensor cores.
        dict(name="eim_f32_1m_d2_k25", method="eim", dtype="f32", sweep="f32", shape="gau", clusters=25, n=1_000_000,
             d=2, k=25),
        dict(name="eim_f32_8m_d64_k1024", method="eim", dtype="f32", sweep="f32", shape="gau", clusters=100,
             n=8_000_000, d=64, k=1024),
        # A serving loop: 4,096 independent instances (n from 1,000 to 200,000,
        # d in {3, 8, 32}, k from 8 to 128), planned once and replayed.
        dict(name="batch_bf16_4096", method="plan", dtype="f32", sweep="bf16", count=4096, mix=1000, nlo=1_000,
             nhi=200_000),
    ]


# ---------------------------------------------------------------- further cases

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: the method, its sizes (log-uniform, odd ones among them),
    the point set and, where there is one, the sweep."""
    method = rng.choice(["gon"] * 8 + ["radius"] * 4 + ["mrg"] * 3 + ["eim"] * 2 + ["batch", "plan", "plan"])
    if method in ("batch", "plan"):
        return dict(method=method, dtype="f32", sweep=rng.choice(["f32", "bf16"]), count=_log(rng, 16, 2048),
                    mix=rng.randrange(1 << 20), nlo=rng.choice([500, 1_000, 4_000]), nhi=rng.choice([20_000, 200_000]))
    c = dict(method=method, dtype="f32")
    d = rng.choice([_log(rng, 2, 100), rng.choice([2, 3, 8, 10, 16, 32, 64])])
    if method == "eim":   # its rounds need n well above k n^eps ln n
        n = _log(rng, 100_000, 2_000_000)
        k = _log(rng, 2, 50)
    else:
        n = _log(rng, 2_000, min(10_000_000, 500_000_000 // d))
        k = min(_log(rng, 2, 1024), n // 8)
    if method != "eim" and rng.random() < 0.2:
        c["dtype"] = "i32"
    shape = "unif" if c["dtype"] == "i32" else rng.choice(["unif", "gau", "unb"])
    c.update(shape=shape, n=n, d=d, k=k)
    if shape != "unif":
        c["clusters"] = rng.choice([10, 25, 50, 100])
    if method != "radius":
        c["sweep"] = "f32" if c["dtype"] == "i32" else rng.choice(["f32", "f32", "bf16", "fp16"])
    if method == "mrg":
        c["m"] = min(_log(rng, 2, 200), max(2, n // (2 * k)))
        c["zipf"] = rng.choice([0.0, 1.1])
    return c


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _mixture(n, d, clusters, sigma, lo, hi, heavy, gen):
    """Gaussian clusters; `heavy` of the points go to cluster 0."""
    means = lo + (hi - lo) * torch.rand(clusters, d, generator=gen, device=DEV)
    comp = torch.randint(0, clusters, (n,), generator=gen, device=DEV)
    if heavy > 0.0:
        comp[torch.rand(n, generator=gen, device=DEV) < heavy] = 0
    x = torch.randn(n, d, generator=gen, device=DEV).mul_(sigma)
    return x.add_(means[comp])


def _int_hi(d):
    """Largest coordinate for which d * hi^2 stays below 2^32 (at most 1023)."""
    return min(1023, int(math.sqrt((2.0 ** 32 - 1) / d)))


def _points(case, gen):
    n, d = case["n"], case["d"]
    if case["dtype"] == "i32":
        return torch.randint(0, _int_hi(d) + 1, (n, d), generator=gen, device=DEV, dtype=torch.int32)
    if case["shape"] == "unif":   # the unit box; the 2-D sets on [0, 100)^2
        x = torch.rand(n, d, generator=gen, device=DEV)
        return x.mul_(100.0) if d == 2 else x
    heavy = 0.5 if case["shape"] == "unb" else 0.0
    if d == 2:
        return _mixture(n, d, case["clusters"], 0.1, 0.0, 100.0, heavy, gen)
    return _mixture(n, d, case["clusters"], 0.5 if d >= 16 else 1.0, -10.0 if d >= 16 else -50.0,
                    10.0 if d >= 16 else 50.0, heavy, gen)


def _sizes(case):
    """(n, d, k, shape) of every instance of a batch."""
    r = random.Random(case["mix"])
    return [(_log(r, case["nlo"], case["nhi"]), r.choice((3, 8, 32)), r.randint(8, 128),
             r.choice(("unif", "gau", "unb"))) for _ in range(case["count"])]


def _instances(case, gen):
    out = []
    for n, d, _, shape in _sizes(case):
        if shape == "unif":
            out.append(torch.rand(n, d, generator=gen, device=DEV))
        else:
            out.append(_mixture(n, d, 25, 0.1, 0.0, 1.0, 0.9 if shape == "unb" else 0.0, gen))
    return out


def _offsets(case):
    """MRG part boundaries (a CPU tensor), or None for the balanced split."""
    if not case["zipf"]:
        return None
    m, n = case["m"], case["n"]
    w = [i ** -case["zipf"] for i in range(1, m + 1)]
    size = [max(1, int(n * v / sum(w))) for v in w]
    size[0] += n - sum(size)
    off = [0]
    for s in size:
        off.append(off[-1] + s)
    return torch.tensor(off, dtype=torch.int64)


def prepare(case, seed):
    """The points on the GPU, and the plan or center set the program keeps."""
    gen = _gen(seed)
    s = dict(case=case, seed=seed)
    if case["method"] in ("batch", "plan"):
        s["x"] = _instances(case, gen)
        s["k"] = [k for _, _, k, _ in _sizes(case)]
        if case["method"] == "plan":
            s["plan"] = kc.kc_batch_plan_create(s["x"], s["k"], sweep=case["sweep"])
        return s
    s["x"] = _points(case, gen)
    if case["method"] == "radius":
        s["centers"] = _center_set(case, gen)
    if case["method"] == "mrg":
        s["offsets"] = _offsets(case)
    return s


def _center_set(case, gen):
    """Distinct center indices drawn at random, as a seeding would pick them."""
    n, k = case["n"], case["k"]
    step = n // k
    return torch.arange(k, device=DEV) * step + torch.randint(0, step, (k,), generator=gen, device=DEV)


# ---------------------------------------------------------------- one pass

def run(state):
    case, x = state["case"], state["x"]
    m = case["method"]
    if m == "plan":
        kc.kc_batch_plan_run(state["plan"])
        p = state["plan"]
        return [torch.cat(p.centers), p.k_out, p.radii]
    if m == "batch":
        r = kc.kc_gonzalez_batch(x, state["k"], sweep=case["sweep"])
        return [torch.cat([g.centers for g in r]), torch.tensor([g.k_out for g in r], dtype=torch.int32),
                torch.tensor([g.radius for g in r], dtype=torch.float64)]
    if m == "radius":
        r = kc.kc_radius(x, state["centers"])
        return [r.argmax, r.radius]
    if m == "gon":
        g = kc.kc_gonzalez(x, case["k"], sweep=case["sweep"])
    elif m == "mrg":
        g = kc.kc_mrg(x, case["k"], case["m"], state["offsets"], sweep=case["sweep"])
    else:
        g = kc.kc_eim(x, case["k"], eps=EPS, phi=PHI, seed=state["seed"], sweep=case["sweep"])
    return [g.centers, g.k_out, g.radius]


# ---------------------------------------------------------------- what it is

def work(case):
    """Each point read once and each output written once; operations are those
    of the distance evaluations that define the method, 3 d each (subtract,
    multiply, add): k n for GON and the radius, k |part| and k |union| for MRG,
    the first sampling round's |R| |S| for EIM."""
    if case["method"] in ("batch", "plan"):
        sz = _sizes(case)
        return {"bytes": sum(4 * n * d + 8 * k + 12 for n, d, k, _ in sz), "flops": sum(3 * n * d * k for n, d, k, _ in sz)}
    n, d, k = case["n"], case["d"], case["k"]
    pairs = n * k
    if case["method"] == "mrg":
        pairs += case["m"] * k * k + n * k
    elif case["method"] == "eim":
        pairs += n * min(n, 9 * k * n ** EPS * math.log(n))
    return {"bytes": 4 * n * d + 8 * k + 12, "flops": 3 * pairs * d}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------- in 64 bits

def _canonical(acc, t):
    """fma(t, t, acc) of float32 values: the product is exact in float64."""
    t = t.double()
    return torch.addcmul(acc.double(), t, t).float()


def _dist(xT, c):
    """Canonical squared distances of the points (columns of xT, or of
    [.., n] slices) to c, as order-preserving int64 value bits."""
    if xT.dtype == torch.int32:
        acc = torch.zeros((), dtype=torch.int64, device=DEV)
        for j in range(xT.shape[0]):
            t = xT[j].long() - c[j].long()
            acc = acc + t * t
        return acc
    acc = torch.zeros((), dtype=torch.float32, device=DEV)
    for j in range(xT.shape[0]):
        acc = _canonical(acc, xT[j] - c[j])
    return acc.view(torch.int32).long()


def _gon(xT, k):
    """Center indices of GON from point 0 (xT: [d, n])."""
    n = xT.shape[1]
    low = 0xFFFFFFFF - torch.arange(n, device=DEV)
    got, m = [torch.zeros((), dtype=torch.int64, device=DEV)], None
    while len(got) < min(k, n):
        v = _dist(xT, xT[:, got[-1]])
        m = v if m is None else torch.minimum(m, v)
        got.append(0xFFFFFFFF - ((m << 32 | low).max() & 0xFFFFFFFF))
    return torch.stack(got)


def _far(x, c):
    """(index, distance) of the point farthest from its nearest center, float64."""
    c, best, at = c.double(), [], []
    rows = max(1, (1 << 24) // c.shape[0])
    for i in range(0, x.shape[0], rows):
        p = x[i:i + rows].double()
        s = torch.zeros(p.shape[0], c.shape[0], dtype=torch.float64, device=DEV)
        for j in range(x.shape[1]):
            t = p[:, j, None] - c[None, :, j]
            s += t * t
        v = s.amin(1)
        best.append(v.amax())
        at.append(i + torch.nonzero(v == best[-1])[0, 0])
    b = torch.stack(best)
    w = torch.nonzero(b == b.amax())[0, 0]
    return int(at[w]), math.sqrt(float(b[w]))


def _mix(z):
    z = (z ^ (z >> 30 & (1 << 34) - 1)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ (z >> 27 & (1 << 37) - 1)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ (z >> 31 & (1 << 33) - 1)


def _uniform(seed, it, x, stream):
    z = seed + (((it << 33) | (x << 1) | stream) + 1) * (0x9E3779B97F4A7C15 - (1 << 64))
    return (_mix(z) >> 11 & (1 << 53) - 1).double() * 2.0 ** -53


def _near(xT, sT):
    """Nearest canonical distance of each column of xT to the columns of sT."""
    out = []
    for i in range(0, xT.shape[1], max(1, (1 << 26) // sT.shape[1])):
        out.append(_dist(xT[:, i:i + max(1, (1 << 26) // sT.shape[1]), None], sT[:, None, :]).amin(1))
    return torch.cat(out)


def _eim(x, k, seed):
    n = x.shape[0]
    base = n ** EPS * math.log(n)
    xT = x.t().contiguous()
    R, S, it = torch.arange(n, device=DEV), torch.zeros(0, dtype=torch.int64, device=DEV), 0
    while R.numel() > 4.0 / EPS * k * base:
        new = _uniform(seed, it, R, 0) < min(1.0, 9.0 * k * base / R.numel())
        H = R[_uniform(seed, it, R, 1) < min(1.0, 4.0 * base / R.numel())]
        S = torch.cat([S, R[new]])
        if H.numel() and S.numel():
            key = (_near(xT[:, H], xT[:, S]) << 32 | 0xFFFFFFFF - H).sort(descending=True).values
            p = min(H.numel(), max(1, math.ceil(PHI * math.log(n))))
            R = R[_near(xT[:, R], xT[:, S]) > (key[p - 1] >> 32)]
        else:
            R = R[~new]
        it += 1
    C = torch.unique(torch.cat([S, R]))
    return C[_gon(xT[:, C], k)]


def exact(case, seed):
    """The same outputs from plain torch: selections by their definition on the
    canonical float32 distance, radii in float64."""
    gen = _gen(seed)
    m = case["method"]
    if m in ("batch", "plan"):
        sz = _sizes(case)
        if sum(k * (d + 4) for _, d, k, _ in sz) > 300_000:
            return None   # too many small steps
        xs = _instances(case, gen)
        cs = [_gon(x.t().contiguous(), k) for x, (_, _, k, _) in zip(xs, sz)]
        return [torch.cat(cs), torch.tensor([c.numel() for c in cs], dtype=torch.int32),
                torch.tensor([_far(x, x[c])[1] for x, c in zip(xs, cs)], dtype=torch.float64)]
    n, d, k = case["n"], case["d"], case["k"]
    x = _points(case, gen)
    if m == "radius":
        return list(_far(x, x[_center_set(case, gen)]))
    if m == "gon":
        c = _gon(x.t().contiguous(), k)
    elif m == "mrg":
        off = _offsets(case)
        off = [i * n // case["m"] for i in range(case["m"] + 1)] if off is None else off.tolist()
        if case["m"] * k * (d + 4) > 400_000:
            return None   # too many small steps
        u = torch.cat([a + _gon(x[a:b].t().contiguous(), k) for a, b in zip(off, off[1:])]).sort().values
        c = u[_gon(x[u].t().contiguous(), k)]
    else:
        if n * 9 * k * n ** EPS * math.log(n) * d > 2e11:
            return None   # the first round's pairs alone take over 20 seconds
        c = _eim(x, k, seed)
    return [c, c.numel(), _far(x, x[c])[1]]
