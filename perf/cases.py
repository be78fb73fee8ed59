"""What the library is timed on: its sweeps, batches and walkers as a program
calls them, from one small lattice to the largest workloads.

A case is a dict of plain values.  ``prepare`` builds the lattice, batch or
walker set with its start state on the GPU, ``run`` makes one call of the kind
a simulation repeats (it continues the chain, so it can be called again),
``work`` counts the bytes and lane operations one such call cannot do without
and ``exact`` repeats the first call of a fresh state in FP64 with plain torch.

Lattice outputs are the energy and |m| series and the whole configuration
after the call, written into a device tensor.  Continuous spins start around a
common axis, as after a cold start's first sweeps, so |m| is well above its
rounding.
"""
import math

import numpy as np
import torch

from paper_1107_5463_gb300 import inputs, spinmc

EA_SIDES = (8, 12, 16, 24, 32)


def listed():
    return [
        # the paper-sized small lattice, E and |m| every sweep, a long series per call
        dict(name="ising2d_L64", kind="lattice", n=1, d=2, L=64, rule="metropolis",
             storage="i8", bonds=False, sweeps=1000, measure=False),
        # the largest workload: 2.7e8 byte spins at the critical point, out of L2
        dict(name="ising2d_L16384", kind="lattice", n=1, d=2, L=16384, rule="metropolis",
             storage="i8", bonds=False, sweeps=8, measure=False),
        # a finite-size-scaling series is not made of multiples of 32
        dict(name="ising2d_L1000", kind="lattice", n=1, d=2, L=1000, rule="metropolis",
             storage="i8", bonds=False, sweeps=100, measure=False),
        # multispin-coded storage of the 3D workload, resident in L2
        dict(name="ising3d_L512_bits", kind="lattice", n=1, d=3, L=512, rule="metropolis",
             storage="bits", bonds=False, sweeps=8, measure=False),
        # one +-J disorder sample, a few sweeps between measurements: the smallest call
        dict(name="ea3d_L20", kind="lattice", n=1, d=3, L=20, rule="metropolis",
             storage="i8", bonds=True, sweeps=10, measure=True),
        # the FP32 workloads: unit vectors out of L2, angles in L2
        dict(name="heis3d_L256", kind="lattice", n=3, d=3, L=256, rule="metropolis",
             storage="f32", bonds=False, sweeps=8, measure=False),
        dict(name="xy2d_L4096", kind="lattice", n=2, d=2, L=4096, rule="metropolis",
             storage="f32", bonds=False, sweeps=8, measure=False),
        # the XY model in three dimensions, an ordinary side
        dict(name="xy3d_L100", kind="lattice", n=2, d=3, L=100, rule="metropolis",
             storage="f32", bonds=False, sweeps=16, measure=False),
        # the other local rule: von Mises draws by rejection
        dict(name="xy2d_L4096_heatbath", kind="lattice", n=2, d=2, L=4096, rule="heatbath",
             storage="f32", bonds=False, sweeps=4, measure=False),
        # cluster updates at the critical point, large clusters present
        dict(name="sw2d_L8192", kind="lattice", n=1, d=2, L=8192, rule="sw",
             storage="i8", bonds=False, sweeps=4, measure=False),
        # mixed-side spin-glass samples with replica exchange in one launch
        dict(name="ea3d_batch", kind="batch", d=3, samples=512, temps=32, sweeps=20),
        # Wang-Landau walkers in narrow windows over the whole energy range: each call
        # starts again at ln f = 1 and refines the estimates so far
        dict(name="wl2d_L64", kind="walkers", rule="wl", L=64, wpw=128, sweeps=10),
    ]


def _log_even(rng, lo, hi):
    return 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)


def draw(rng):
    what = rng.choice(["ising", "ising", "small", "bits", "ea", "heis", "xy", "xy3d", "xyhb", "sw",
                       "batch", "walkers"])
    if what == "batch":
        return dict(kind="batch", d=rng.choice([2, 3, 3]), samples=rng.randint(16, 512),
                    temps=rng.choice([8, 20, 32, 32]), sweeps=rng.randint(4, 20))
    if what == "walkers":
        L = rng.choice([16, 32, 64])
        return dict(kind="walkers", rule=rng.choice(["wl", "muca"]), L=L,
                    wpw=rng.choice([32, 64, 96, 128]), sweeps=rng.randint(2, 8))
    c = dict(kind="lattice", n=1, d=rng.choice([2, 3]), rule="metropolis", storage="i8",
             bonds=False, measure=rng.random() < 0.3)
    most = 5.0e8   # site updates of one call
    if what == "small":
        c["L"] = _log_even(rng, 16, 256) if c["d"] == 2 else _log_even(rng, 8, 40)
        most = 2.0e7
    elif what == "ising":
        c["L"] = _log_even(rng, 256, 12000) if c["d"] == 2 else _log_even(rng, 40, 480)
    elif what == "bits":
        c["storage"] = "bits"
        c["L"] = 64 * rng.randint(2, 200) if c["d"] == 2 else 64 * rng.randint(1, 8)
    elif what == "ea":
        c["bonds"] = True
        c["L"] = _log_even(rng, 16, 1024) if c["d"] == 2 else _log_even(rng, 8, 96)
        most = 1.0e8
    elif what == "heis":
        c.update(n=3, storage="f32")
        c["L"] = _log_even(rng, 200, 3000) if c["d"] == 2 else _log_even(rng, 40, 240)
        most = 1.0e8
    elif what in ("xy", "xy3d", "xyhb"):
        c.update(n=2, storage="f32", d=3 if what == "xy3d" else 2)
        c["rule"] = "heatbath" if what == "xyhb" else "metropolis"
        c["L"] = _log_even(rng, 200, 4000) if c["d"] == 2 else _log_even(rng, 40, 240)
        most = 6.0e7
    else:
        c["rule"] = "sw"
        c["L"] = _log_even(rng, 64, 6000) if c["d"] == 2 else _log_even(rng, 16, 300)
        most = 1.5e8
    n_most = max(2, min(1000, int(most / c["L"] ** c["d"])))
    c["sweeps"] = max(2, round(math.exp(rng.uniform(math.log(2), math.log(n_most)))))
    return c


def beta_of(c):
    if c["n"] == 1:
        if c["bonds"]:
            return 0.9
        return inputs.BETA_C_2D_ISING if c["d"] == 2 else inputs.BETA_3D_ISING
    if c["n"] == 2:
        return 1.12 if c["d"] == 2 else 0.5
    return inputs.BETA_3D_HEISENBERG if c["d"] == 3 else 1.5


def start_spins(c, seed):
    """Continuous start configuration around a common axis, on the GPU (FP32)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    N = c["L"] ** c["d"]
    if c["n"] == 2:
        a = torch.randn(N, generator=g, device="cuda") * 0.7 + 2.5
        return torch.remainder(a, 2.0 * math.pi).clamp_(0.0, 6.2831850)
    v = torch.randn((N, 3), generator=g, device="cuda")
    v[:, 2] += 1.5
    return v / v.norm(dim=1, keepdim=True)


def bonds_of(c, seed):
    """+-1 forward bonds (d, N) of one disorder sample, on the GPU."""
    g = torch.Generator(device="cuda").manual_seed(seed + 77)
    b = torch.randint(0, 2, (c["d"], c["L"] ** c["d"]), generator=g, device="cuda",
                      dtype=torch.int8)
    return 2 * b - 1


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        sides = inputs.ea_sample_sizes(c["samples"], EA_SIDES)
        b = spinmc.Batch(c["d"], sides, c["temps"], inputs.geometric_betas(c["temps"]), seed=seed)
        return dict(case=c, seed=seed, b=b)
    if c["kind"] == "walkers":
        N, width = c["L"] ** 2, 4
        klo = np.arange(0, N - width + 1, width).astype(np.int32)
        w = spinmc.Walkers(c["L"], klo, klo + width, c["wpw"], seed=seed)
        # multicanonical weights -ln(number of states), Gaussian in the energy
        E = 4.0 * (klo[:, None] + np.arange(w.kmax)[None, :]) - 2.0 * N
        return dict(case=c, seed=seed, w=w, lnW=E * E / (4.0 * N))
    storage = spinmc.SL_STORE_BITS if c["storage"] == "bits" else None
    lat = spinmc.Lattice(c["d"], c["L"], n=c["n"], seed=seed, storage=storage,
                         J_bonds=bonds_of(c, seed) if c["bonds"] else None)
    if c["n"] > 1:
        spinmc.sl_set_spins(lat.h, start_spins(c, seed))
        out = torch.empty((lat.N,) if c["n"] == 2 else (lat.N, 3), dtype=torch.float32,
                          device="cuda")
    else:
        out = torch.empty(lat.N, dtype=torch.int8, device="cuda")
    if c["rule"] == "heatbath":
        lat.set_update(spinmc.SL_UPDATE_HEATBATH)
    if c["rule"] == "sw":
        lat.set_update(spinmc.SL_UPDATE_SW)
        lat.sweep(beta_of(c), 12, seed + 5)  # towards equilibrium: large clusters
    return dict(case=c, seed=seed, lat=lat, beta=beta_of(c), out=out)


def run(state):
    c, seed = state["case"], state["seed"]
    if c["kind"] == "batch":
        return {"E": state["b"].run(c["sweeps"], seed + 1, series=True)}
    if c["kind"] == "walkers":
        w = state["w"]
        if c["rule"] == "wl":
            spinmc.sl_walkers_write(w.h, stage=np.zeros(w.nwalk, np.int32))
            w.wl(c["sweeps"], final_stage=20, seed=seed + 1)
        else:
            w.muca(state["lnW"], c["sweeps"], seed=seed + 1)
        S, H, level, stage, visited = w.read()
        return {"S": S, "H": H.view(np.int32), "level": level, "stage": stage,
                "visited": visited.view(np.int64)}
    lat = state["lat"]
    E, m = lat.sweep_series(state["beta"], c["sweeps"], seed + 1)
    got = {"E": E, "absm": m, "spins": state["out"]}
    if c["measure"]:
        got["E_now"], got["M_now"] = lat.measure()
    spinmc.sl_get_spins(lat.h, state["out"])
    return got


def work(case):
    """Bytes: the state read and written once (and couplings, outputs);
    flops: 32-bit lane operations of the updates, the Philox call first."""
    c = case
    if c["kind"] == "batch":
        sites = sum(L ** c["d"] for L in inputs.ea_sample_sizes(c["samples"], EA_SIDES))
        return {"bytes": sites * (2 * c["temps"] / 8 + c["d"] / 8) + 8 * c["samples"] *
                c["sweeps"] * c["temps"], "flops": 28 * sites * c["temps"] * c["sweeps"]}
    if c["kind"] == "walkers":
        N = c["L"] ** 2
        nwalk = (N // 4) * c["wpw"]
        return {"bytes": nwalk * (2 * N / 8 + 2 * 5 * 12),
                "flops": (40 if c["rule"] == "wl" else 36) * nwalk * N * c["sweeps"]}
    N = c["L"] ** c["d"]
    site = {1: 1.0 if c["storage"] == "i8" else 0.125, 2: 4.0, 3: 12.0}[c["n"]]
    nat = {1: 1.0, 2: 4.0, 3: 12.0}[c["n"]]
    ops = {1: 28, 2: 100 if c["rule"] == "heatbath" else 66, 3: 115}[c["n"]]
    return {"bytes": N * (2 * site + nat + (c["d"] if c["bonds"] else 0)) + 16 * c["sweeps"],
            "flops": ops * N * c["sweeps"]}


# ------------------------------------------------ the same call in FP64 ----

MASK = 0xFFFFFFFF


def philox(c0, t, c3, seed):
    """Philox4x32-10 of counters (c0, t, 0, c3) keyed by seed: four int64 tensors."""
    def halves(m, v):
        p = m * v  # wraps mod 2^64
        return (p >> 32) & MASK, p & MASK
    k0, k1 = seed & MASK, (seed >> 32) & MASK
    x, y, z, w = c0, torch.full_like(c0, t), torch.zeros_like(c0), torch.full_like(c0, c3)
    for _ in range(10):
        h0, l0 = halves(0xD2511F53, x)
        h1, l1 = halves(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return x, y, z, w


def u24(x):
    return (x >> 8).double() * 2.0 ** -24


class Colours:
    """Checkerboard halves of a natural-order lattice as arrays [..., W]: the
    site at column k of a row with parity p sits at x = 2k + p."""

    def __init__(self, d, L):
        self.d, self.L, self.W = d, L, L // 2
        y = torch.arange(L, device="cuda")
        row = y if d == 2 else y[:, None] + y[None, :]
        self.par = [((row + c) & 1).bool()[..., None] for c in range(2)]

    def split(self, a):
        """a: (N, ...) natural order -> the two colour arrays."""
        v = a.reshape((self.L,) * (self.d - 1) + (self.W, 2) + a.shape[1:])
        ax = self.d  # the pair axis
        e, o = v.select(ax, 0), v.select(ax, 1)
        sh = self.par[0].shape + (1,) * (a.dim() - 1)
        p = self.par[0].reshape(sh)
        return [torch.where(p, o, e), torch.where(p, e, o)]

    def join(self, a0, a1):
        sh = self.par[0].shape + (1,) * (a0.dim() - self.d)
        p = self.par[0].reshape(sh)
        v = torch.stack([torch.where(p, a1, a0), torch.where(p, a0, a1)], dim=self.d)
        return v.reshape((self.L ** self.d,) + a0.shape[self.d:])

    def neighbours(self, c, b):
        """The values of b (colour 1 - c) at the neighbours -x, +x, -y, +y (-z, +z)
        of the sites of colour c."""
        p = self.par[c].reshape(self.par[c].shape + (1,) * (b.dim() - self.d))
        ax = self.d - 1
        out = [torch.where(p, b, b.roll(1, ax)), torch.where(p, b.roll(-1, ax), b)]
        for k in range(self.d - 1):
            out += [b.roll(1, ax - 1 - k), b.roll(-1, ax - 1 - k)]
        return out


def best_fisher(h, beta, angle, j, t, c, seed):
    """Heat-bath angles: the von Mises rejection method, FP64."""
    kappa = beta * h.norm(dim=-1)
    tau = 1 + torch.sqrt(1 + 4 * kappa * kappa)
    s2 = torch.sqrt(2 * tau)
    rho = 2 * kappa / (tau + s2)
    gfac, cnum = (1 - rho) / (1 + rho), (tau + s2) * (1 - rho * rho) ** 2 / 4
    base = torch.atan2(h[..., 1], h[..., 0])
    todo = torch.arange(j.numel(), device="cuda")
    shape, angle = angle.shape, angle.reshape(-1).clone()
    for a in range(32):
        if todo.numel() == 0:
            break
        jj = j[todo]
        o = philox(jj >> 1, t, a << 16 | c, seed)
        odd = (jj & 1).bool()
        o1, U2 = torch.where(odd, o[2], o[0]), u24(torch.where(odd, o[3], o[1]))
        wv = math.pi / 2 * u24(o1)
        r, cw = rho.reshape(-1)[todo], torch.cos(wv)
        cc = cnum.reshape(-1)[todo] / ((1 - r) ** 2 + 4 * r * cw * cw)
        ok = (cc * (2 - cc) > U2) | (torch.log(cc / U2) + 1 - cc >= 0)
        delta = 2 * torch.atan2(gfac.reshape(-1)[todo] * torch.sin(wv), cw)
        delta = torch.where((o1 & 1).bool(), -delta, delta)
        th = torch.remainder(base.reshape(-1)[todo] + delta, 2 * math.pi)
        angle[todo[ok]] = th[ok]
        todo = todo[~ok]
    return angle.reshape(shape)


def exact(case, seed):
    c = case
    if c["kind"] != "lattice" or c["rule"] == "sw":
        return None  # whole numbers: energies, counts, fixed-point ln g, spins
    if c["L"] ** c["d"] * c["sweeps"] > 4.0e9 or c["sweeps"] > 4000:
        return None
    geo, beta, sw_seed, d, L, n = Colours(c["d"], c["L"]), beta_of(c), seed + 1, c["d"], c["L"], c["n"]
    H = L ** d // 2
    shape = (L,) * (d - 1) + (L // 2,)
    j = torch.arange(H, device="cuda")
    if n == 1:
        # the start configuration: +1 iff the top bit of the site's output is set
        grp = torch.arange((H + 3) // 4, device="cuda")
        S = []
        for col in range(2):
            o = torch.stack(philox(grp, 0, 2 | col, seed), 1).reshape(-1)[:H]
            S.append(torch.where((o >> 31).bool(), 1, -1).to(torch.int8).reshape(shape))
        B = [geo.split(b) for b in bonds_of(c, seed)] if c["bonds"] else None
    else:
        a = start_spins(c, seed).double()
        S = geo.split(a)
        if n == 2:
            A, S = S, [torch.stack([torch.cos(s), torch.sin(s)], -1) for s in S]

    def field(col):
        nb = geo.neighbours(col, S[1 - col])
        if n == 1 and B is not None:
            # backward neighbours own their bond, forward bonds are the site's
            for mu in range(d):
                back = geo.neighbours(col, B[mu][1 - col])[2 * mu]
                nb[2 * mu], nb[2 * mu + 1] = nb[2 * mu] * back, nb[2 * mu + 1] * B[mu][col]
        h = nb[0].clone()
        for v in nb[1:]:
            h += v
        return h

    E, m = [], []
    for t in range(c["sweeps"]):
        for col in range(2):
            h = field(col)
            if n == 1:
                o = torch.stack(philox(grp, t, col, sw_seed), 1).reshape(-1)[:H].reshape(shape)
                sh = S[col] * h
                lim = torch.tensor([math.exp(-beta * 2.0 * k) * 2.0 ** 32 if k > 0 else 2.0 ** 33
                                    for k in range(-2 * d, 2 * d + 1)],
                                   dtype=torch.float64, device="cuda")
                flip = o.double() < lim[(sh + 2 * d).int()]
                S[col] = torch.where(flip, -S[col], S[col])
                del o, flip
            elif c["rule"] == "heatbath":
                A[col] = best_fisher(h, beta, A[col], j, t, col, sw_seed)
                S[col] = torch.stack([torch.cos(A[col]), torch.sin(A[col])], -1)
            else:
                if n == 2:
                    o = philox(j >> 1, t, col, sw_seed)
                    odd = (j & 1).bool()
                    u, th = u24(torch.where(odd, o[2], o[0])), 2 * math.pi * u24(
                        torch.where(odd, o[3], o[1]))
                    new = torch.stack([torch.cos(th), torch.sin(th)], -1)
                else:
                    o = philox(j, t, col, sw_seed)
                    u, z, ph = u24(o[0]), 2 * u24(o[1]) - 1, 2 * math.pi * u24(o[2])
                    r = torch.sqrt((1 - z) * (1 + z))
                    new = torch.stack([r * torch.cos(ph), r * torch.sin(ph), z], -1)
                new, u = new.reshape(shape + (n,)), u.reshape(shape)
                dE = -((new - S[col]) * h).sum(-1)
                acc = (dE <= 0) | (u < torch.exp(-beta * dE))
                S[col] = torch.where(acc[..., None], new, S[col])
                if n == 2:
                    A[col] = torch.where(acc, th.reshape(shape), A[col])
                elif (t + 1) % 16 == 0:
                    S[col] = S[col] / S[col].norm(dim=-1, keepdim=True)
        h = field(1)
        if n == 1:
            E.append(-float((S[1].int() * h.int()).sum()))
            M = [float(S[0].sum(dtype=torch.int64) + S[1].sum(dtype=torch.int64))]
        else:
            E.append(-float((S[1] * h).sum()))
            M = (S[0] + S[1]).reshape(-1, n).sum(0).tolist()
        m.append(math.sqrt(sum(v * v for v in M)) / L ** d)
    got = {"E": np.array(E), "absm": np.array(m), "spins": geo.join(*(A if n == 2 else S))}
    if c["measure"]:
        got["E_now"], got["M_now"] = E[-1], np.array(M + [m[-1]])
    return got
