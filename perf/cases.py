"""The work that users of this library have it do, as measurable cases.

Every case goes through the public Python calls (``Plan``, ``Batch``,
``refine_noise``, ``autograd``). ``listed()`` names the cases, ``draw(rng)``
makes further ones of the same ranges, ``prepare`` builds what a program holds
before the call, ``run`` is one pass and ``work`` its compulsory bytes and
operations. ``exact`` evaluates the same definitions in 64 bits with plain
torch: the Philox4x32-10 / Box-Muller noise, Eqs. 1-3, the Sec. 2.4 merge and
degrading, the Appendix A refinement, the cloud-in-cell loss and the shell
estimator.
"""
import math

import numpy as np
import torch

import paper_2511_10353_gb300 as gg
from paper_2511_10353_gb300 import autograd as gga

COSMOS = {"bbks": gg.workloads.BBKS, "eh_nw": gg.workloads.EH_NW}
DTYPES = {"f32": torch.float32, "f64": torch.float64}


def _zeldovich(name, n, box, z, prec, outputs, cosmo="bbks", given=False, gas=False):
    return {"name": name, "op": "zeldovich", "n": n, "box": box, "z": z, "prec": prec,
            "outputs": outputs, "cosmo": cosmo, "given": given, "gas": gas}


def listed():
    return [
        # the smallest run in use: one 64^3 box in double precision, all outputs
        # (a parameter scan or a unit test of a simulation code); launches count
        _zeldovich("zeldovich_64_f64", 64, 100.0, 50.0, "f64", "psi+pos+vel"),
        # a density field from the caller's noise on a grid that is no power of two
        {"name": "field_96_f32", "op": "field", "n": 96, "box": 96.0, "z": 50.0, "prec": "f32",
         "cosmo": "bbks", "given": True},
        # the headline: particles of one single-precision 512^3 box from a seed
        _zeldovich("zeldovich_512_f32", 512, 500.0, 100.0, "f32", "pos+vel"),
        # the same box in double precision
        _zeldovich("zeldovich_512_f64", 512, 500.0, 100.0, "f64", "pos+vel"),
        # a large production box on the most common large grid
        _zeldovich("zeldovich_1024_f32", 1024, 1000.0, 100.0, "f32", "pos+vel"),
        # the largest: the displacement fields of the 1536^3 parent box
        _zeldovich("displacement_1536_f32", 1536, 2000.0, 100.0, "f32", "psi", "eh_nw"),
        # an ensemble: independent realizations of uneven sizes in one call
        {"name": "ensemble_16", "op": "batch", "count": 16, "sizes": "128,192,256,384", "z": 50.0},
        # one step of a constrained-realization fit: loss and its gradient
        {"name": "fit_512", "op": "loss", "n": 512, "box": 500.0, "z": 100.0, "prec": "f32",
         "density": "cic", "targets": 4096, "radius": 8.0},
        # white noise of the next resolution level (Appendix A)
        {"name": "refine_768_1536", "op": "refine", "n": 768, "kind": "2", "prec": "f32"},
        # fine particles that take their large scales from the coarse level (Sec. 2.4)
        {"name": "merge_256_512", "op": "merge", "n": 512, "n_low": 256, "box": 500.0, "z": 100.0,
         "prec": "f32"},
        # a velocity field brought down to a coarser grid (Sec. 2.4)
        {"name": "degrade_512_256", "op": "degrade", "n": 256, "r": 2, "box": 500.0, "prec": "f32"},
        # the statistics that are printed for a field: P(k) and moments (Sec. 2.1)
        {"name": "diagnose_512", "op": "diagnose", "n": 512, "box": 500.0, "prec": "f32"},
    ]


def _sizes(lo, hi, r=1):
    """The even grids 2^a 3^b in [lo, hi] whose r-fold refinement is wanted too,
    without those whose strided copies the library did not lay out on 128-byte
    boundaries when these ranges were drawn up."""
    out, left_out = set(), (324, 486, 972)
    for a in range(1, 13):
        for b in range(0, 8):
            v = 2 ** a * 3 ** b
            if lo <= v <= hi and v not in left_out and r * v not in left_out:
                out.add(v)
    return sorted(out)


def _pick(rng, sizes):
    """One of ``sizes``, spread over their logarithm."""
    x = math.exp(rng.uniform(math.log(sizes[0]), math.log(sizes[-1])))
    return min(sizes, key=lambda s: abs(math.log(s / x)))


def draw(rng):
    op = rng.choice(["zeldovich", "zeldovich", "zeldovich", "field", "batch", "loss", "refine",
                     "merge", "degrade", "diagnose"])
    # redshifts of initial conditions (a particle on the box edge may land on either
    # side of it after one rounding, which later redshifts would show too often)
    z = float(rng.choice([20, 30, 50, 100]))
    cosmo = rng.choice(["bbks", "eh_nw"])
    prec = "f64" if rng.random() < 0.25 else "f32"
    if op == "zeldovich":
        n = _pick(rng, _sizes(32, 384 if prec == "f64" else 1024))
        gas = rng.random() < 0.2
        outputs = "pos+vel" if gas else rng.choice(["pos+vel", "pos+vel", "psi", "psi+pos+vel"])
        c = _zeldovich("", n, round(n * rng.uniform(0.5, 2.0), 3), z, prec, outputs, cosmo,
                       rng.random() < 0.3, gas)
        del c["name"]
        return c
    if op == "field":
        n = _pick(rng, _sizes(24, 384 if prec == "f64" else 864))
        return {"op": op, "n": n, "box": round(n * rng.uniform(0.5, 2.0), 3), "z": z, "prec": prec,
                "cosmo": cosmo, "given": rng.random() < 0.5}
    if op == "batch":
        k = rng.randint(2, 4)
        sizes = sorted(rng.sample([64, 96, 128, 144, 192, 256, 288, 384], k))
        return {"op": op, "count": rng.randint(k, 14), "sizes": ",".join(map(str, sizes)), "z": z}
    if op == "loss":
        n = _pick(rng, _sizes(48, 432))
        return {"op": op, "n": n, "box": float(n), "z": z, "prec": prec if n <= 216 else "f32",
                "density": rng.choice(["cic", "linear"]), "targets": rng.randint(100, 4096),
                "radius": round(rng.uniform(4.0, 12.0), 3)}
    if op == "refine":
        n = 6 * int(round(math.exp(rng.uniform(math.log(8), math.log(112 if prec == "f32" else 48)))))
        return {"op": op, "n": n, "kind": rng.choice(["hr", "3/2", "2", "2", "2-linear", "2-sine", "4/3"]),
                "prec": prec}
    if op == "merge":
        r = rng.choice([2, 3])
        n_low = _pick(rng, _sizes(24, (384 if prec == "f32" else 128) // r, r))
        return {"op": op, "n": r * n_low, "n_low": n_low, "box": float(r * n_low), "z": z, "prec": prec}
    if op == "degrade":
        r = rng.choice([2, 2, 3, 4])
        n = _pick(rng, _sizes(24, (768 if prec == "f32" else 384) // r))
        return {"op": op, "n": n, "r": r, "box": float(n), "prec": prec}
    n = _pick(rng, _sizes(32, 640 if prec == "f32" else 288))
    return {"op": "diagnose", "n": n, "box": round(n * rng.uniform(0.5, 2.0), 3), "prec": prec}


# ------------------------------------------------------------------- inputs
# Made by torch alone, so that prepare() and exact() see the same values.
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _white(n, dtype, gen):
    return torch.randn((n, n, n), dtype=dtype, device="cuda", generator=gen)


def _modes(n, lo=0, hi=None):
    """Integer frequencies of the rfftn layout, x rows lo .. hi - 1 (int64)."""
    m = torch.arange(n, device="cuda")
    m = torch.where(m < n // 2, m, m - n)
    return m[lo:hi, None, None], m[None, :, None], torch.arange(n // 2 + 1, device="cuda")[None, None, :]


def _smooth_field(n, dtype, gen):
    """A displacement-like random field: white noise with its small scales damped."""
    f = torch.fft.rfftn(_white(n, torch.float32, gen))
    mx, my, mz = _modes(n)
    f /= 1.0 + (mx * mx + my * my + mz * mz).float() / 64.0
    return (3.0 * torch.fft.irfftn(f, s=(n, n, n))).to(dtype)


def _fit_inputs(case, seed):
    n, gen, dtype = case["n"], _gen(seed), DTYPES[case["prec"]]
    noise = _white(n, dtype, gen)
    targets = torch.randint(0, n ** 3, (case["targets"],), device="cuda", generator=gen)
    return noise, targets, torch.randn(case["targets"], dtype=dtype, device="cuda", generator=gen)


def _batch_specs(case):
    sizes = [int(s) for s in case["sizes"].split(",")]
    return [dict(n=n, box=float(n), cosmo=gg.workloads.BBKS, z_init=case["z"], prec="f32")
            for n in (sizes[i % len(sizes)] for i in range(case["count"]))]


def _plan(case, n=None):
    return gg.Plan(n or case["n"], case["box"], COSMOS[case.get("cosmo", "bbks")], case.get("z", 50.0),
                   case["prec"])


# -------------------------------------------------------------------- cases
def prepare(case, seed):
    op, s = case["op"], {"case": case, "op": case["op"], "seed": int(seed)}
    if op == "batch":
        specs = _batch_specs(case)
        s["batch"] = gg.Batch(specs)
        s["seeds"] = [int(seed) + i for i in range(len(specs))]
        # pos and vel of each realization in one allocation
        s["grids"] = [torch.empty((2, 3) + (w["n"],) * 3, device="cuda") for w in specs]
        s["out"] = {"psi": None, "pos": [list(g[0]) for g in s["grids"]],
                    "vel": [list(g[1]) for g in s["grids"]]}
        return s
    n, dtype = case["n"], DTYPES[case["prec"]]
    if op == "refine":
        s["parent"] = _white(n, dtype, _gen(seed))
        s["out"] = torch.empty(gg.refine_dims(n, case["kind"]), dtype=dtype, device="cuda")
        return s
    s["plan"] = plan = _plan(case)
    if op == "zeldovich":
        s["noise"] = _white(n, dtype, _gen(seed)) if case["given"] else None
        want = case["outputs"].split("+")
        s["out"] = {k: [plan.empty() for _ in range(3)] if k in want else [None] * 3
                    for k in ("psi", "pos", "vel")}
        if case["gas"]:
            s["out"]["pos_gas"] = [plan.empty() for _ in range(3)]
    elif op == "field":
        s["noise"] = _white(n, dtype, _gen(seed)) if case["given"] else None
        s["out"] = plan.empty()
    elif op == "loss":
        s["noise"], s["targets"], s["y"] = _fit_inputs(case, seed)
        s["noise"].requires_grad_(True)
    elif op == "merge":
        gen = _gen(seed)
        s["coarse"] = _plan(case, case["n_low"])
        s["psi_low"] = [_smooth_field(case["n_low"], dtype, gen) for _ in range(3)]
        s["noise"] = _white(n, dtype, gen)
        s["large"] = [s["coarse"].empty() for _ in range(3)]
        s["out"] = {"psi": [None] * 3, "pos": [plan.empty() for _ in range(3)],
                    "vel": [plan.empty() for _ in range(3)]}
    elif op == "degrade":
        s["high"] = _smooth_field(case["n"] * case["r"], dtype, _gen(seed))
        s["out"] = plan.empty()
    elif op == "diagnose":
        s["field"] = _white(n, dtype, _gen(seed))
    return s


def run(s):
    op, case = s["op"], s["case"]
    if op == "batch":
        s["batch"].run(s["seeds"], s["out"])
        return s["grids"]
    if op == "refine":
        return gg.refine_noise(s["parent"], s["seed"], case["kind"], out=s["out"])
    plan = s["plan"]
    if op == "zeldovich":
        if case["gas"]:
            return plan.zeldovich_gas(0.16, seed=s["seed"], noise=s["noise"], out=s["out"])
        return plan.zeldovich(seed=s["seed"], noise=s["noise"], out=s["out"])
    if op == "field":
        return plan.gaussian_field(seed=s["seed"], noise=s["noise"], out=s["out"])
    if op == "loss":
        loss = gga.smoothed_density_loss(s["noise"], plan, s["targets"], s["y"], radius=case["radius"],
                                         density=case["density"])
        return {"loss": loss.detach(), "grad": torch.autograd.grad(loss, s["noise"])[0]}
    if op == "merge":
        r_s = 2.0 * case["box"] / case["n_low"]
        large = [s["coarse"].large_scales(f, r_s, out=o) for f, o in zip(s["psi_low"], s["large"])]
        return {"large": large,
                "out": plan.zeldovich_merge(large, r_s, noise=s["noise"], out=s["out"])}
    if op == "degrade":
        return plan.degrade(s["high"], out=s["out"])
    return {"power": plan.power_spectrum(s["field"]), "moments": plan.moments(s["field"])}


def work(case):
    """Inputs read once and outputs written once; 2.5 n log2 n per real transform."""
    op = case["op"]

    def ffts(n, count):
        return 2.5 * n ** 3 * 3 * math.log2(n) * count

    if op == "batch":
        ns = [w["n"] for w in _batch_specs(case)]
        return {"bytes": sum(24 * n ** 3 for n in ns), "flops": sum(ffts(n, 4) for n in ns)}
    n, size = case["n"], 8 if case["prec"] == "f64" else 4
    cells = n ** 3
    if op == "refine":
        nl, nh, _, _ = _refine_kind(case["kind"])
        child = (n // nl * nh) ** 3
        return {"bytes": size * (cells + child), "flops": 6 * nh * child}
    if op == "zeldovich":
        outs = 3 * (len(case["outputs"].split("+")) + (1 if case["gas"] else 0))
        return {"bytes": size * cells * (outs + (1 if case["given"] else 0)), "flops": ffts(n, 4)}
    if op == "field":
        return {"bytes": size * cells * (2 if case["given"] else 1), "flops": ffts(n, 2)}
    if op == "loss":
        return {"bytes": size * 2 * cells, "flops": ffts(n, 12 if case["density"] == "cic" else 8)}
    if op == "merge":
        low = case["n_low"] ** 3
        return {"bytes": size * (7 * cells + 6 * low), "flops": ffts(n, 4) + ffts(case["n_low"], 6)}
    if op == "degrade":
        return {"bytes": size * 2 * cells, "flops": ffts(n, 2)}
    return {"bytes": size * cells, "flops": ffts(n, 1) + 8 * cells}


# ------------------------------------------- the same definitions in 64 bits
def _philox(seed, first, count):
    """Words of the groups first .. first + count - 1 (int64 tensors in [0, 2^32))."""
    mask = 0xFFFFFFFF
    g = torch.arange(first, first + count, dtype=torch.int64, device="cuda")
    c = [g & mask, g >> 32, torch.zeros_like(g), torch.zeros_like(g)]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(m, x):  # 32 x 32 -> (high, low); a product past 2^63 wraps, its bits stay right
        p = x * m
        return (p >> 32) & mask, p & mask

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _noise_cells(seed, lo, hi):
    """W of the cells lo .. hi - 1 by the two-output Box-Muller map."""
    first = lo >> 2
    w = _philox(int(seed), first, ((hi + 3) >> 2) - first)
    out = torch.empty((w[0].numel(), 4), dtype=torch.float64, device="cuda")
    for p in (0, 2):
        rho = torch.sqrt(-2.0 * torch.log((w[p].double() + 1.0) * 2.0 ** -32))
        ang = w[p + 1].double() * (2.0 * math.pi * 2.0 ** -32)
        out[:, p], out[:, p + 1] = rho * torch.cos(ang), rho * torch.sin(ang)
    return out.reshape(-1)[lo - 4 * first:hi - 4 * first]


def _noise_grid(seed, n):
    out = torch.empty(n ** 3, dtype=torch.float64, device="cuda")
    step = 1 << 25
    for lo in range(0, n ** 3, step):
        hi = min(n ** 3, lo + step)
        out[lo:hi] = _noise_cells(seed, lo, hi)
    return out.reshape(n, n, n)


def _gauss_nodes(edges, order=24):
    """Composite Gauss-Legendre nodes and weights on the pieces between edges."""
    x, w = np.polynomial.legendre.leggauss(order)
    mid, half = 0.5 * (edges[1:] + edges[:-1]), 0.5 * (edges[1:] - edges[:-1])
    return (mid[:, None] + half[:, None] * x).ravel(), (half[:, None] * w).ravel()


class _Cosmology:
    """P(k), D and the velocity factor in 64 bits (flat, sigma_8-normalised)."""

    def __init__(self, p):
        self.om, self.h, self.ns, self.p = p["omega_m"], p["h"], p["n_s"], p
        ln, w = _gauss_nodes(np.linspace(math.log(1e-6), math.log(0.05), 200))
        k, wk = _gauss_nodes(np.linspace(0.05, 1000.0, 8001))
        k, w = np.concatenate([np.exp(ln), k]), np.concatenate([w * np.exp(ln), wk])
        x = 8.0 * k
        top = np.where(x < 1e-2, 1.0 - x * x / 10.0 + x ** 4 / 280.0,
                       3.0 * (np.sin(x) - x * np.cos(x)) / np.maximum(x, 1e-9) ** 3)
        self.amp = p["sigma_8"] ** 2 / (np.sum(w * k * k * self._shape(k) * top * top) / (2 * math.pi ** 2))

    def _shape(self, k):
        p = self.p
        if p["tf"] == "bbks":
            q = k / (self.om * self.h)
            t = np.log1p(2.34 * q) / (2.34 * q) * (
                1.0 + 3.89 * q + (16.1 * q) ** 2 + (5.46 * q) ** 3 + (6.71 * q) ** 4) ** -0.25
        else:
            om_h2, ob_h2, fb = self.om * self.h ** 2, p["omega_b"] * self.h ** 2, p["omega_b"] / self.om
            s = 44.5 * math.log(9.83 / om_h2) / math.sqrt(1.0 + 10.0 * ob_h2 ** 0.75)
            al = 1.0 - 0.328 * math.log(431.0 * om_h2) * fb + 0.38 * math.log(22.3 * om_h2) * fb * fb
            gam = self.om * self.h * (al + (1.0 - al) / (1.0 + (0.43 * k * self.h * s) ** 4))
            q = k * (p["t_cmb"] / 2.7) ** 2 / gam
            l0 = np.log(2.0 * math.e + 1.8 * q)
            t = l0 / (l0 + (14.2 + 731.0 / (1.0 + 62.5 * q)) * q * q)
        return k ** self.ns * t * t

    def _e2(self, a):
        return self.om / a ** 3 + 1.0 - self.om

    def _du(self, a):  # (5 Om / 2) E int_0^a da / (a E)^3, with a = u^2
        u, w = _gauss_nodes(np.linspace(0.0, math.sqrt(a), 65))
        x = u * u
        f = 2.0 * u * (x / (self.om + (1.0 - self.om) * x ** 3)) ** 1.5
        return 2.5 * self.om * math.sqrt(self._e2(a)) * np.sum(w * f)

    def growth(self, z):
        return self._du(1.0 / (1.0 + z)) / self._du(1.0)

    def velocity(self, z):
        a = 1.0 / (1.0 + z)
        e2 = self._e2(a)
        f = -3.0 * self.om / a ** 3 / (2.0 * e2) + 5.0 * self.om / (2.0 * a * a * e2 * self._du(a))
        return 100.0 * a * math.sqrt(e2) * f

    def density_filter(self, n, box, z):
        """D sqrt(P / V) N^-3/2 by m^2 (0 at k = 0), on the GPU."""
        k = 2.0 * math.pi / box * np.sqrt(np.arange(1, 3 * (n // 2) ** 2 + 1, dtype=np.float64))
        s = self.growth(z) * np.sqrt(self.amp * self._shape(k) / box ** 3) / float(n) ** 1.5
        return torch.from_numpy(np.concatenate([[0.0], s])).cuda()


def _slabs(n):
    step = max(1, (1 << 26) // (n * n))
    return [(lo, min(n, lo + step)) for lo in range(0, n, step)]


def _scaled(spec, n, factor):
    """``spec`` times factor(mx, my, mz, m2) with the |m_j| = N/2 modes dropped (new tensor)."""
    out = torch.empty_like(spec)
    for lo, hi in _slabs(n):
        mx, my, mz = _modes(n, lo, hi)
        keep = (mx != -(n // 2)) & (my != -(n // 2)) & (mz != n // 2)
        f = factor(mx, my, mz, mx * mx + my * my + mz * mz)
        out[lo:hi] = torch.where(keep, spec[lo:hi] * f, 0.0)
    return out


def _real(spec, n):
    return torch.fft.irfftn(spec, s=(n, n, n), norm="forward")


def _psi(spec, n, box, table, j, cut=0):
    """psi_j from the unnormalised spectrum of the noise; modes with m2 < cut dropped."""
    def factor(mx, my, mz, m2):
        mj = (mx, my, mz)[j].double() * (box / (2.0 * math.pi))
        f = table[m2] * mj / m2.clamp(min=1).double()
        return 1j * torch.where(m2 >= cut, f, 0.0)
    return _real(_scaled(spec, n, factor), n)


def _particles(psi, n, box, j, vfac, extra=0.0):
    sh = [1, 1, 1]
    sh[j] = n
    q = ((torch.arange(n, device="cuda").double() + 0.5) * (box / n) + extra).reshape(sh)
    return torch.remainder(q + psi, box), vfac * psi


def _refine_kind(kind):
    r2, r3, r6, r7, r20 = (math.sqrt(v) for v in (2, 3, 6, 7, 20))
    one, two = [[1.0]], [[1 / r2, 1 / r2], [-1 / r2, 1 / r2]]
    three = [[1 / r3] * 3, [-1 / r2, 0.0, 1 / r2], [-1 / r6, 2 / r6, -1 / r6]]
    even = [0.5, 0.5, 0.5, 0.5], [-0.5, 0.5, 0.5, -0.5]
    four = [even[0], [-r7 / 4, -0.25, 0.25, r7 / 4], even[1], [0.25, -r7 / 4, r7 / 4, -0.25]]
    linear = [even[0], [-3 / r20, -1 / r20, 1 / r20, 3 / r20], even[1], [1 / r20, -3 / r20, 3 / r20, -1 / r20]]
    sine = [even[0], [-0.5, -0.5, 0.5, 0.5], even[1], [0.5, -0.5, 0.5, -0.5]]
    return {"hr": (1, 2, one, two), "3/2": (2, 3, two, three), "2": (2, 4, two, four),
            "2-linear": (2, 4, two, linear), "2-sine": (2, 4, two, sine),
            "4/3": (3, 4, three, four)}[kind]


def _exact_refine(case, seed):
    n, (nl, nh, f, e) = case["n"], _refine_kind(case["kind"])
    parent = _white(n, DTYPES[case["prec"]], _gen(seed))
    p = n // nl
    nc = p * nh
    f = torch.tensor(f, dtype=torch.float64, device="cuda")
    e = torch.tensor(e, dtype=torch.float64, device="cuda")
    out = torch.empty((nc, nc, nc), dtype=torch.float64, device="cuda")

    def along(a, m, d):  # contract dimension d of a with the rows of m
        return torch.movedim(torch.tensordot(a, m, dims=([d], [1])), -1, d)

    for i in range(p):  # one layer of patches along x at a time
        a = _noise_cells(int(seed), i * nh * nc * nc, (i + 1) * nh * nc * nc).reshape(nh, p, nh, p, nh)
        v = parent[i * nl:(i + 1) * nl].double().reshape(nl, p, nl, p, nl)
        a[:nl, :, :nl, :, :nl] = along(along(along(v, f, 0), f, 2), f, 4)
        out[i * nh:(i + 1) * nh] = along(along(along(a, e.T, 0), e.T, 2), e.T, 4).reshape(nh, nc, nc)
    return out


def _exact_fit(case, seed):
    n, box, radius = case["n"], case["box"], case["radius"]
    noise, targets, y = _fit_inputs(case, seed)
    w = noise.double().requires_grad_(True)
    cosmo = _Cosmology(gg.workloads.BBKS)
    table = cosmo.density_filter(n, box, case["z"])
    mx, my, mz = _modes(n)
    m2 = mx * mx + my * my + mz * mz
    keep = ((mx != -(n // 2)) & (my != -(n // 2)) & (mz != n // 2)).double()
    delta_k = torch.fft.rfftn(w) * (table[m2] * keep)
    if case["density"] == "cic":
        cell, i0, frac = box / n, [], []
        over = box / (2.0 * math.pi) / m2.clamp(min=1).double()
        for j, m in enumerate((mx, my, mz)):
            psi = _real(delta_k * (1j * m.double() * over), n)
            sh = [1, 1, 1]
            sh[j] = n
            u = torch.arange(n, device="cuda").double().reshape(sh) + psi / cell
            low = torch.floor(u.detach())
            i0.append(low.long() % n)
            frac.append(u - low)
            del psi, u, low
        delta = torch.full((n ** 3,), -1.0, dtype=torch.float64, device="cuda")
        for corner in range(8):
            wt, idx = 1.0, 0
            for j in range(3):
                hi = (corner >> (2 - j)) & 1
                wt = wt * (frac[j] if hi else 1.0 - frac[j])
                idx = idx * n + (i0[j] + hi) % n
            delta = delta.index_add(0, idx.reshape(-1), wt.reshape(-1))
            del wt, idx
        delta = delta.reshape(n, n, n)
    else:
        delta = _real(delta_k, n)
    k2 = (2.0 * math.pi / box) ** 2 * m2.double()
    ds = torch.fft.irfftn(torch.fft.rfftn(delta) * (torch.exp(-0.5 * k2 * radius * radius) * keep), s=(n, n, n))
    res = ds.reshape(-1)[targets] - y.double()
    loss = (res * res).sum()
    return {"loss": loss.detach(), "grad": torch.autograd.grad(loss, w)[0]}


def _exact_merge(case, seed):
    n, nl, box, gen, dtype = case["n"], case["n_low"], case["box"], _gen(seed), DTYPES[case["prec"]]
    low = [_smooth_field(nl, dtype, gen) for _ in range(3)]
    noise = _white(n, dtype, gen)
    r_s = 2.0 * box / nl
    cut = math.ceil((box / (2.0 * math.pi * r_s)) ** 2)
    sinc = lambda m: torch.sinc(m.double() / nl) ** 2  # noqa: E731
    large = [torch.fft.irfftn(_scaled(torch.fft.rfftn(v.double()), nl, lambda mx, my, mz, m2: torch.where(
        m2 < cut, 1.0 / (sinc(mx) * sinc(my) * sinc(mz)), 0.0)), s=(nl, nl, nl)) for v in low]
    u = (torch.arange(n, device="cuda").double() + 0.5) * nl / n - 0.5
    first = torch.floor(u)
    t, i0 = u - first, first.long() % nl
    i1 = (i0 + 1) % nl
    cosmo = _Cosmology(gg.workloads.BBKS)
    table, vfac = cosmo.density_filter(n, box, case["z"]), cosmo.velocity(case["z"])
    spec = torch.fft.rfftn(noise.double())
    out = {"psi": [None] * 3, "pos": [], "vel": []}
    for j in range(3):
        c = large[j]
        for d in range(3):  # linear between cell centres, one axis after the other
            sh = [1, 1, 1]
            sh[d] = n
            tt = t.reshape(sh)
            c = c.index_select(d, i0) * (1.0 - tt) + c.index_select(d, i1) * tt
        pos, vel = _particles(c + _psi(spec, n, box, table, j, cut), n, box, j, vfac)
        out["pos"].append(pos)
        out["vel"].append(vel)
    return {"large": large, "out": out}


def _exact_degrade(case, seed):
    n, r = case["n"], case["r"]
    g = _smooth_field(n * r, DTYPES[case["prec"]], _gen(seed))[::r, ::r, ::r].double()
    t = 2.0 * math.pi * (r - 1) / (2.0 * r) / n
    spec = _scaled(torch.fft.rfftn(g), n, lambda mx, my, mz, m2: torch.polar(
        torch.ones_like(m2, dtype=torch.float64), t * (mx + my + mz).double()))
    return torch.fft.irfftn(spec, s=(n, n, n))


def _exact_diagnose(case, seed):
    n, box, nb = case["n"], case["box"], case["n"] // 2
    f = _white(n, DTYPES[case["prec"]], _gen(seed)).double()
    spec = torch.fft.rfftn(f)
    sums = torch.zeros((3, nb), dtype=torch.float64, device="cuda")
    edges = (2 * torch.arange(1, nb + 1, device="cuda") - 1) ** 2  # shell b starts at 4 m2 = (2b - 1)^2
    for lo, hi in _slabs(n):
        mx, my, mz = _modes(n, lo, hi)
        m2 = mx * mx + my * my + mz * mz
        keep = (mx != -(n // 2)) & (my != -(n // 2)) & (mz != n // 2)
        b = torch.searchsorted(edges, 4 * m2, right=True)
        keep = keep & (b < nb)
        wt = torch.where(mz == 0, 1.0, 2.0).double().expand(m2.shape)[keep]
        for i, v in enumerate((wt, wt * m2[keep].double().sqrt(), wt * spec[lo:hi][keep].abs().square())):
            sums[i] += torch.bincount(b[keep], weights=v, minlength=nb)
    cnt, mag, power = sums.cpu().numpy()
    safe = np.maximum(cnt, 1.0)
    mean = f.mean()
    return {"power": (2.0 * math.pi / box * mag / safe, box ** 3 / float(n) ** 6 * power / safe, None),
            "moments": (float(mean), float((f - mean).square().mean()), float(f.min()), float(f.max()))}


def exact(case, seed):
    op = case["op"]
    if op == "refine":
        return _exact_refine(case, seed)
    if op == "loss":
        return _exact_fit(case, seed)
    if op == "merge":
        return _exact_merge(case, seed)
    if op == "degrade":
        return _exact_degrade(case, seed)
    if op == "diagnose":
        return _exact_diagnose(case, seed)
    if op == "batch":
        cosmo, out = _Cosmology(gg.workloads.BBKS), []
        for i, w in enumerate(_batch_specs(case)):
            n, box = w["n"], w["box"]
            table, vfac = cosmo.density_filter(n, box, case["z"]), cosmo.velocity(case["z"])
            spec = torch.fft.rfftn(_noise_grid(int(seed) + i, n))
            pv = [_particles(_psi(spec, n, box, table, j), n, box, j, vfac) for j in range(3)]
            out.append(torch.stack([torch.stack([v[0] for v in pv]), torch.stack([v[1] for v in pv])]))
        return out
    n, box, z = case["n"], case["box"], case["z"]
    cosmo = _Cosmology(COSMOS[case["cosmo"]])
    table = cosmo.density_filter(n, box, z)
    noise = _white(n, DTYPES[case["prec"]], _gen(seed)).double() if case["given"] else _noise_grid(seed, n)
    spec = torch.fft.rfftn(noise)
    del noise
    if op == "field":
        return _real(_scaled(spec, n, lambda mx, my, mz, m2: table[m2]), n)
    vfac, want = cosmo.velocity(z), case["outputs"].split("+")
    out = {k: [None] * 3 for k in ("psi", "pos", "vel") + (("pos_gas",) if case["gas"] else ())}
    for j in range(3 if n <= 1024 else 1):  # of the largest grid the first component alone
        psi = _psi(spec, n, box, table, j)
        half = 0.5 * box / n
        pos, vel = _particles(psi, n, box, j, vfac, -0.16 * half if case["gas"] else 0.0)
        for k, v in (("psi", psi), ("pos", pos), ("vel", vel)):
            out[k][j] = v if k in want else None
        if case["gas"]:
            out["pos_gas"][j] = _particles(psi, n, box, j, vfac, 0.84 * half)[0]
        del psi, pos, vel
    return out
