"""What this library is asked to do, as cases that can be timed and compared.

Every case is a gap-filling call of the public binding on synthetic data of the kind the method is
studied on: a Gaussian field N(50, 10^2) with exponential covariance exp(-kappa |h|), a fraction p
of whose sites is removed at random. Five kinds of call:

``job``     the whole method from host arrays to a host prediction, ``GapFiller(z, mask).fill``:
            creation, temperature tuning, equilibration, sampling, prediction, release.
``chain``   a handle that a program keeps: ``run(equil, samples)`` at a known temperature, then the
            prediction into a device tensor; for FP64 functions also the energy of the state.
``bounded`` the same with bounded Metropolis proposals whose width adapts.
``batch``   many uneven problems in one launch, tuned, equilibrated, sampled; their predictions.
``energy``  the bond energy of a state that the caller holds on the device.
"""
import math

import numpy as np
import torch

import paper_1910_08448_gb300 as mpr

TWO_PI = 2.0 * math.pi
KAPPA = 0.2        # decay of the synthetic field's covariance
WORK_T = 0.065     # about what the tuning finds for these fields (p = 0.9, kappa = 0.2)


def _chain(name, Lx, Ly, p, setup, equil, samples, acc="f64"):
    return {"name": name, "kind": "chain", "Lx": Lx, "Ly": Ly, "p": p, "setup": setup, "acc": acc,
            "equil": equil, "samples": samples}


def listed():
    return [
        # the smallest study size, whole job: thousands of sweeps of 4096 sites, launches and
        # latency; the default options (FP32 spins and functions, FP64 energy)
        {"name": "job 64 SDS", "kind": "job", "Lx": 64, "Ly": 64, "p": 0.33, "setup": "SDS",
         "equil": 1000, "samples": 100},
        # a user's odd-sized grid, host arrays in and out, 16-bit spins
        {"name": "job 777x523 HDS", "kind": "job", "Lx": 777, "Ly": 523, "p": 0.66,
         "setup": "HDS", "equil": 200, "samples": 50},
        # a small map with few gaps, many sweeps
        _chain("chain 256 SDS", 256, 256, 0.33, "SDS", 400, 100),
        # the middle study size
        _chain("chain 1024 SDS", 1024, 1024, 0.66, "SDS", 200, 20),
        # the massive-data size of the benchmark, FP16 spins: ten plain sweeps to one sampled, as
        # in the benchmark's 2000 + 200
        _chain("chain 4096 HDS", 4096, 4096, 0.9, "HDS", 100, 10),
        # the largest study size: FP32 spins that no cache holds; 5 plain sweeps to one sampled
        _chain("chain 16384 SDS", 16384, 16384, 0.9, "SDS", 20, 4),
        # BF16 spins, FP32 compensated sums, a rectangular grid whose tiles are all ragged
        _chain("chain 2501x1333 BDS Kahan", 2501, 1333, 0.66, "BDS", 100, 20, acc="kahan"),
        # adapted bounded proposals: the acceptance is counted and the width moved every sweep
        {"name": "bounded 2048 HDS", "kind": "bounded", "Lx": 2048, "Ly": 2048, "p": 0.9,
         "setup": "HDS", "width": 6.0, "target": 0.4, "equil": 100, "samples": 10},
        # the double-precision side of every precision comparison, at the benchmark's size
        _chain("chain 4096 DDD", 4096, 4096, 0.9, "DDD", 4, 2),
        # double precision on a small odd grid with few gaps (a reference run next to an FP32 one)
        _chain("chain 321x257 DSD", 321, 257, 0.33, "DSD", 12, 6),
        # many uneven problems at once, tuned: sides log-uniform on 64 ... 1024
        {"name": "batch 48 HDS", "kind": "batch", "n": 48, "shapes": 4, "L_max": 1024,
         "setup": "HDS", "equil": 500, "samples": 100},
        # a diagnostic on a state that another program holds on the device
        {"name": "energy 4096", "kind": "energy", "Lx": 4096, "Ly": 4096, "q": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi):
    """Two sides with a geometric mean log-uniform on [lo, hi] and an aspect up to 3."""
    L, a = _log_int(rng, lo, hi), math.exp(rng.uniform(-0.55, 0.55))
    return max(lo // 2, int(round(L * a))), max(lo // 2, int(round(L / a)))


def draw(rng):
    kind = rng.choice(["job", "chain", "chain", "chain", "bounded", "double", "double", "batch", "energy"])
    p = rng.choice([0.33, 0.66, 0.9])
    if kind == "job":
        Lx, Ly = _sides(rng, 48, 768)
        return {"kind": "job", "Lx": Lx, "Ly": Ly, "p": p,
                "setup": rng.choice(["SDS", "SSS", "HDS", "BDS", "HDH"]),
                "equil": rng.randint(100, 400), "samples": rng.randint(10, 60)}
    if kind in ("chain", "bounded"):
        Lx, Ly = _sides(rng, 64, 8192)
        n = max(10, min(400, int(2e9 / (Lx * Ly))))
        c = {"kind": kind, "Lx": Lx, "Ly": Ly, "p": p,
             "setup": rng.choice(["SDS", "SSS", "HDS", "HSS", "BDS"] if kind == "bounded" else
                                 ["SDS", "SDS", "SSS", "HDS", "HDS", "HSS", "BDS", "HDH", "DDS"]),
             "equil": n, "samples": max(2, n // 10)}
        if kind == "bounded":
            return dict(c, width=rng.uniform(0.5, 6.0), target=rng.choice([0.0, 0.4]))
        return dict(c, acc=rng.choice(["f64", "f64", "kahan"]))
    if kind == "double":
        Lx, Ly = _sides(rng, 64, 2048)
        return {"kind": "chain", "Lx": Lx, "Ly": Ly, "p": p, "setup": rng.choice(["DDD", "DSD"]),
                "acc": "f64", "equil": rng.randint(2, 8), "samples": rng.randint(1, 3)}
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(6, 48), "shapes": rng.randrange(1 << 20),
                "L_max": rng.choice([256, 512, 768]), "setup": rng.choice(["HDS", "SDS", "BDS"]),
                "equil": rng.randint(100, 500), "samples": rng.randint(10, 100)}
    Lx, Ly = _sides(rng, 64, 8192)
    return {"kind": "energy", "Lx": Lx, "Ly": Ly, "q": rng.choice([0.5, 0.5, 1.0, 0.3])}


# --- inputs -----------------------------------------------------------------------------------

def _field(Lx, Ly, gen, kappa=KAPPA):
    """N(50, 10^2) with covariance 100 exp(-kappa |h|) on the torus, (Ly, Lx) float64 on the GPU."""
    def lag(n):
        i = torch.arange(n, device="cuda", dtype=torch.float32)
        return torch.minimum(i, n - i)
    r = torch.sqrt(lag(Ly)[:, None] ** 2 + lag(Lx)[None, :] ** 2)
    lam = torch.fft.rfft2(100.0 * torch.exp(-kappa * r)).real.clamp_(min=0.0)
    w = torch.fft.rfft2(torch.randn((Ly, Lx), device="cuda", generator=gen))
    z = torch.fft.irfft2(w * lam.sqrt(), s=(Ly, Lx))
    return (50.0 + z).double().contiguous()


def _data(Lx, Ly, p, seed, kappa=KAPPA):
    """A field and its mask (1 = measured) on the GPU, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    z = _field(Lx, Ly, gen, kappa)
    mask = (torch.rand((Ly, Lx), device="cuda", generator=gen) >= p).to(torch.uint8)
    mask[0, :2] = 1   # a tiny grid keeps one measured pair
    return z, mask


def _shapes(case):
    """The batch's problems: (Lx, Ly, p, kappa), as many as case["n"]."""
    rng = np.random.default_rng(case["shapes"])
    out = []
    for _ in range(case["n"]):
        L = math.exp(rng.uniform(math.log(64), math.log(case["L_max"])))
        a = math.exp(rng.uniform(-math.log(4.0), math.log(4.0)))
        out.append((int(round(L * math.sqrt(a))), int(round(L / math.sqrt(a))),
                    float(rng.choice([0.33, 0.66, 0.9])), float(rng.uniform(0.05, 0.5))))
    return out


class _Batch:
    """Releases its batch when the program drops it."""

    def __init__(self, b, n):
        self.b, self.n = b, n

    def __del__(self):
        mpr.mpr_batch_destroy(self.b)


def _chain_seed(seed):
    return 1000 + seed


def prepare(case, seed):
    kind = case["kind"]
    if kind == "job":
        z, mask = _data(case["Lx"], case["Ly"], case["p"], seed)
        return {"case": case, "seed": seed, "z": z.cpu().numpy(), "mask": mask.cpu().numpy()}
    if kind in ("chain", "bounded"):
        z, mask = _data(case["Lx"], case["Ly"], case["p"], seed)
        f = mpr.GapFiller(z, mask, setup=case["setup"], seed=_chain_seed(seed),
                          acc=case.get("acc", "f64"))
        f.set_temperature(WORK_T)
        if kind == "bounded":
            mpr.mpr_set_proposal(f.h, case["width"], case["target"])
        return {"case": case, "filler": f, "out": torch.empty_like(z)}
    if kind == "batch":
        zs, ms = [], []
        for i, (Lx, Ly, p, kappa) in enumerate(_shapes(case)):
            z, mask = _data(Lx, Ly, p, 100003 * (i + 1) + seed, kappa)
            zs.append(z.cpu().numpy())
            ms.append(mask.cpu().numpy())
        b = mpr.mpr_batch_create(zs, ms, case["setup"], seed=_chain_seed(seed))
        return {"case": case, "batch": _Batch(b, case["n"])}
    gen = torch.Generator(device="cuda").manual_seed(seed)
    # a state as a chain leaves it: a smooth field on [0, 2 pi) with thermal noise
    z = _field(case["Lx"], case["Ly"], gen)
    lo, hi = z.min(), z.max()
    noise = 0.3 * torch.randn(z.shape, device="cuda", dtype=torch.float64, generator=gen)
    phi = (TWO_PI * (z - lo) / (hi - lo) + noise).clamp_(0.0, 6.2831)
    return {"case": case, "phi": phi.contiguous(),
            "out": torch.empty(1, dtype=torch.float64, device="cuda")}


# --- the calls --------------------------------------------------------------------------------

def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "job":
        with mpr.GapFiller(state["z"], state["mask"], setup=case["setup"],
                           seed=_chain_seed(state["seed"])) as f:
            zhat = f.fill(case["equil"], case["samples"])
            return {"zhat": zhat, "T": f.T, "e_bond": f.info()["e_bond_mean"]}
    if kind in ("chain", "bounded"):
        f = state["filler"]
        f.run(case["equil"], case["samples"])
        r = {"zhat": f.predict(state["out"]), "e_bond": f.info()["e_bond_mean"]}
        if kind == "bounded":
            r["width"] = mpr.mpr_get_proposal(f.h)
        if case["setup"][2] == "D":
            r["e_state"] = mpr.mpr_energy(f.h)[0]
        return r
    if kind == "batch":
        b = state["batch"]
        T, _ = mpr.mpr_batch_fill(b.b, case["equil"], case["samples"])
        return {"T": T, "zhat": [mpr.mpr_batch_predict(b.b, i) for i in range(b.n)]}
    return mpr.mpr_bond_energy_noalloc(state["phi"], case["q"], state["out"])


# --- what a pass cannot do without --------------------------------------------------------------

STORE_BYTES = {"D": 8, "S": 4, "H": 2, "B": 2}
FLOPS_UPDATE = 150   # one hybrid move: the field, three sine/cosine pairs, exp, atan2, the tests
TUNE_SWEEPS = 2000   # about eight probes of 200 + 50 sweeps


def _sweep_work(sites, p, setup, sweeps, samples):
    """Own colour read, other colour read once, prediction sites written, one mask bit; a sampled
    sweep reads and writes 8 bytes of sums per prediction site."""
    b = STORE_BYTES[setup[0]]
    return (sites * (sweeps * (b * (2 + p) + 0.125) + samples * 16 * p),
            sites * p * sweeps * FLOPS_UPDATE)


def work(case):
    kind = case["kind"]
    if kind == "energy":
        n = case["Lx"] * case["Ly"]
        return {"bytes": 8 * n, "flops": 2 * 30 * n}
    grids = ([(Lx * Ly, p) for Lx, Ly, p, _ in _shapes(case)] if kind == "batch"
             else [(case["Lx"] * case["Ly"], case["p"])])
    sweeps = case["equil"] + case["samples"] + (TUNE_SWEEPS if kind in ("job", "batch") else 0)
    total = [0.0, 0.0]
    for n, p in grids:
        by, fl = _sweep_work(n, p, case["setup"], sweeps, case["samples"])
        total[0] += by + n * (8 + 1 + 8) + (n * (8 + 1) if kind == "job" else 0)
        total[1] += fl
    return {"bytes": total[0], "flops": total[1]}


# --- the same in 64 bits, by plain torch --------------------------------------------------------

def _mulhilo(m, x):
    """High and low words of the 32 x 32 -> 64 bit product (x: int64 tensor below 2^32)."""
    p1, p2 = m * (x & 0xFFFF), m * (x >> 16)
    t = p1 + ((p2 & 0xFFFF) << 16)
    return (p2 >> 16) + (t >> 32), t & 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox-4x32-10; counter words as int64 tensors or numbers, key = seed."""
    x = [c0, c1, c2 + torch.zeros_like(c0), c3]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        h0, l0 = _mulhilo(0xD2511F53, x[0])
        h1, l1 = _mulhilo(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x


def _site_words(X, Y, sweep, tag, seed):
    """The two random words of every site: first drives its proposal, second its acceptance."""
    w = _philox(X >> 2, Y, sweep, (tag << 1) | ((X + Y) & 1), seed)
    second = ((X >> 1) & 1) == 1
    return torch.where(second, w[2], w[0]), torch.where(second, w[3], w[1])


def _exact_chain(case, seed):
    q, T = 0.5, WORK_T
    z, mask = _data(case["Lx"], case["Ly"], case["p"], seed)
    Ly, Lx = z.shape
    frozen = mask != 0
    lo, hi = z[frozen].min(), z[frozen].max()
    Y, X = torch.meshgrid(torch.arange(Ly, device="cuda"), torch.arange(Lx, device="cuda"),
                          indexing="ij")
    key = _chain_seed(seed)
    phi = torch.where(frozen, TWO_PI * ((z - lo) / (hi - lo)),
                      TWO_PI * (_site_words(X, Y, 0, 1, key)[0].double() * 2.0 ** -32))
    colour = (X + Y) & 1

    def field(u):
        h = torch.zeros_like(u)
        h[:, 1:] += u[:, :-1]
        h[:, :-1] += u[:, 1:]
        h[1:] += u[:-1]
        h[:-1] += u[1:]
        return h

    def e_bond(a):
        d = torch.cos(q * (a[:, 1:] - a[:, :-1])).sum() + torch.cos(q * (a[1:] - a[:-1])).sum()
        return -float(d) / (Lx * (Ly - 1) + Ly * (Lx - 1))

    acc = torch.zeros_like(phi)
    energies = []
    for sweep in range(case["equil"] + case["samples"]):
        w_prop, w_acc = _site_words(X, Y, sweep, 0, key)
        prop, u = TWO_PI * (w_prop.double() * 2.0 ** -32), w_acc.double() * 2.0 ** -32
        for c in (0, 1):
            hx, hy = field(torch.cos(q * phi)), field(torch.sin(q * phi))
            dE = ((hx * torch.cos(q * phi) + hy * torch.sin(q * phi))
                  - (hx * torch.cos(q * prop) + hy * torch.sin(q * prop)))
            f1 = torch.where((dE <= 0) | (u < torch.exp(-dE / T)), prop, phi)
            psi = 2.0 * torch.atan2(hy, hx) - q * f1
            r = psi - TWO_PI * torch.floor(psi / TWO_PI)
            fn = torch.where((r <= TWO_PI * q) & ((hx != 0) | (hy != 0)), r / q, f1)
            phi = torch.where((colour == c) & ~frozen, fn, phi)
        if sweep >= case["equil"]:
            acc += phi
            energies.append(e_bond(phi))
    zhat = torch.where(frozen, z, lo + (hi - lo) * (acc / case["samples"] / TWO_PI))
    return {"zhat": zhat, "e_bond": sum(energies) / len(energies), "e_state": e_bond(phi)}


def exact(case, seed):
    if case["kind"] == "energy":
        phi, q = prepare(case, seed)["phi"], case["q"]
        Ly, Lx = phi.shape
        s = torch.cos(q * (phi[:, 1:] - phi[:, :-1])).sum() + torch.cos(q * (phi[1:] - phi[:-1])).sum()
        return (-s / (Lx * (Ly - 1) + Ly * (Lx - 1))).reshape(1)
    if case["kind"] == "chain" and case["setup"][2] == "D":
        return _exact_chain(case, seed)
    # With FP32 functions a proposal near its threshold is decided by FP32 rounding, and the chain
    # goes another way from there: no 64-bit value belongs to these outputs.
    return None
