"""What a user of this framework has it do, as timed calls of its public entry points.

Three kinds of call: one force evaluation at new positions (``forces``), a
short stretch of dynamics from new positions and velocities (``md``), and one
distillation gradient over a batch of labelled frames (``distill``). Sizes and
settings are those of the repository's configurations, tests and benchmark:
water boxes, batched vacuum molecules, periodic replicas and a solvated
polymer, with the 3.5 A small model and the 5.0 A big model, in both precisions.

The networks compute in FP32 (or with BF16 operands) and the library widens
their forces, gradients and energies to FP64 on the way out; the outputs are
returned as the FP32 numbers they are, and positions and velocities as the
single-precision frames that trajectory files hold.
"""
from __future__ import annotations

import json
import math

import numpy as np
import torch

from paper_2510_06562_gb300 import dmts as D
from paper_2510_06562_gb300 import inputs as I

WATER_SITE = 3.105          # A per molecule and axis: 12.42 A for 4, 49.7 A for 16
KB_EV = 8.617333262e-5
ACCEL = 1.602176634e-19 / 1.66053906660e-27 * 1e-10      # eV/(A amu) in A/fs^2
GAMMA_PS, TEMPERATURE = 1.0, 300.0
SEED_SMALL, SEED_BIG = 2, 3  # the models' weights: the repository's


# ------------------------------------------------------------------ the cases
def _water(n_side, stretch=1.0):
    return {"system": "water", "n_side": n_side, "stretch": stretch}


def _md(n_outer, n_inner, dt, single=False, langevin=False):
    return {"kind": "md", "n_outer": n_outer, "n_inner": n_inner, "dt": dt, "single": single, "langevin": langevin}


def listed():
    return [
        # the smallest call: one energy and force of the 192-atom box in the default precision (an
        # optimiser, a scorer or a coupled MD engine that asks for forces one geometry at a time)
        {"name": "forces_water192_fp32", "kind": "forces", **_water(4), "precision": "fp32", "model": "big",
         "virial": False},
        # small-box dynamics with the distilled scheme: every launch and gap counts
        {"name": "md3fs_water192_bf16", **_md(10, 3, 3.0), **_water(4), "precision": "bf16"},
        # single-time-step Langevin dynamics of a 1,536-atom box with the big model alone: how the frames
        # for distillation are sampled, and the reference the distilled scheme is compared with
        {"name": "sts_langevin_water1536_fp32", **_md(10, 1, 1.0, single=True, langevin=True), **_water(8),
         "precision": "fp32"},
        # the headline workload: 12,288-atom water, 3 fs outer / 1 fs inner, tensor-core MLPs
        {"name": "md3fs_water12288_bf16", **_md(10, 3, 3.0), **_water(16), "precision": "bf16"},
        # the same box with the longer outer step, where the small model carries most of the work
        {"name": "md6fs_water12288_bf16", **_md(5, 6, 6.0), **_water(16), "precision": "bf16"},
        # and in the default precision
        {"name": "md3fs_water12288_fp32", **_md(4, 3, 3.0), **_water(16), "precision": "fp32"},
        # energy, forces and virial of the large box in the accuracy-reference precision (pressure, labelling)
        {"name": "forces_virial_water12288_fp32", "kind": "forces", **_water(16), "precision": "fp32",
         "model": "big", "virial": True},
        # 512 independent molecules of 10 to 60 atoms in one launch
        {"name": "md3fs_vacuum512_bf16", **_md(10, 3, 3.0), "system": "vacuum", "n_mol": 512, "precision": "bf16"},
        # labelling a ragged batch of molecules with the big model
        {"name": "forces_vacuum301_fp32", "kind": "forces", "system": "vacuum", "n_mol": 301, "precision": "fp32",
         "model": "big", "virial": False},
        # the largest system: a solvated polymer of about 100,000 atoms and four elements
        {"name": "md3fs_polymer100k_bf16", **_md(3, 3, 3.0), "system": "polymer", "n_heavy": 1000,
         "n_total": 100000, "precision": "bf16"},
        # a training step's gradient on the large box, tensor-core MLPs
        {"name": "distill_water12288_bf16", "kind": "distill", **_water(16), "precision": "bf16", "frames": 8,
         "lambda_e": 1.0},
        # and on a small box of odd size in the default precision
        {"name": "distill_water1029_fp32", "kind": "distill", **_water(7), "precision": "fp32", "frames": 5,
         "lambda_e": 1.0},
    ]


def draw(rng):
    limit = _cost(listed()[9])
    while True:
        case = _draw_once(rng)
        if _cost(case) <= limit:
            return case


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(["forces", "forces", "md", "md", "md", "distill"])
    system = "water" if kind == "distill" else rng.choice(["water", "water", "water", "vacuum", "replicas", "polymer"])
    c = {"kind": kind, "system": system, "precision": rng.choice(["fp32", "bf16"])}
    if system in ("water", "replicas"):
        c["stretch"] = round(rng.uniform(1.0, 1.04), 4)
        c["n_side"] = _log_int(rng, 4, 16 if kind == "distill" else 26) if system == "water" else rng.randint(5, 8)
    if system == "replicas":
        c["n_rep"] = rng.randint(2, 11)
    if system == "vacuum":
        c["n_mol"] = _log_int(rng, 3, 800)
    if system == "polymer":
        c["n_total"] = _log_int(rng, 3000, 80000)
        c["n_heavy"] = c["n_total"] // 100
    if kind == "forces":
        c["model"] = rng.choice(["big", "big", "small"])
        c["virial"] = rng.random() < 0.3
    elif kind == "md":
        if rng.random() < 0.25:
            c.update(_md(rng.randint(1, 12), 1, 1.0, single=True, langevin=rng.random() < 0.4))
        else:
            n = rng.randint(2, 6)
            c.update(_md(rng.randint(1, max(1, 30 // n)), n, float(n), langevin=rng.random() < 0.3))
    else:
        c["frames"] = rng.randint(1, 8)
        c["lambda_e"] = rng.choice([1.0, 0.1])
    return c


# ------------------------------------------------------------------ what a case costs at least
def _atoms_pairs(case):
    """Atoms, and directed pairs within 3.5 and 5.0 A (from the density)."""
    s = case["system"]
    if s == "vacuum":                       # chains of 10 to 60 atoms: mean pair counts of that generator
        n = 35 * case["n_mol"]
        return n, 9.7 * n, 17.6 * n
    n = case["n_total"] if s == "polymer" else 3 * case["n_side"] ** 3 * case.get("n_rep", 1)
    rho = 0.1001 / case.get("stretch", 1.0) ** 3
    return n, n * rho * 4 / 3 * math.pi * 3.5 ** 3, n * rho * 4 / 3 * math.pi * 5.0 ** 3


def _eval_flops(n, pairs, K, F, L):
    """One energy and force: the filter MLP and its derivative once per unordered pair and layer, the
    message products and their adjoints per directed pair, the per-atom MLPs forward and backward."""
    edge = pairs / 2 * 2 * (2 * K * F + 2 * F * F) + pairs * 8 * F
    atom = n * 2 * F * F * (6 * L + 2)
    return L * edge + atom


def work(case):
    n, p_small, p_big = _atoms_pairs(case)
    small = _eval_flops(n, p_small, 8, 32, 1)
    big = _eval_flops(n, p_big, 16, 64, 2)
    weights = 4.0 * (26000 + 6000)
    if case["kind"] == "forces":
        return {"bytes": 48.0 * n + weights, "flops": big if case["model"] == "big" else small}
    if case["kind"] == "md":
        n_small = 0 if case["single"] else case["n_outer"] * case["n_inner"] + 1
        n_big = case["n_outer"] + 1
        return {"bytes": 96.0 * n + weights, "flops": n_small * small + n_big * big}
    # the gradient through the forces: the value and tangent passes and their reverse
    return {"bytes": case["frames"] * 48.0 * n + weights, "flops": case["frames"] * 4 * small}


def _cost(case):
    return work(case)["flops"] * (4.0 if case["precision"] == "fp32" else 1.0)


# ------------------------------------------------------------------ what a user's program has in hand
def _system(case, seed):
    s = case["system"]
    if s == "water":
        n = case["n_side"]
        return I.make_water(n, round(WATER_SITE * n, 2) * case["stretch"], seed)
    if s == "replicas":
        n = case["n_side"]
        box = round(WATER_SITE * n, 2) * case["stretch"]
        return I.replicas([I.make_water(n, box, seed + 1000 * k) for k in range(case["n_rep"])])
    # the same molecules (sizes, elements) at another conformation for every seed
    if s == "vacuum":
        system = I.make_vacuum_batch(case["n_mol"], 10, 60, 0)
    else:
        system = I.make_solvated_polymer(case["n_heavy"], case["n_total"], 1.0, 0)
    system.x = system.x + 0.03 * np.random.default_rng(seed).standard_normal(system.x.shape)
    return system


def _models(n_species):
    sa, ba = I.small_arch(n_species), I.big_arch(n_species)
    return sa, I.init_params(sa, SEED_SMALL), ba, I.init_params(ba, SEED_BIG)


def _frames(case, system, seed):
    """Frames around the structure (0.03 A per component) and their labels by the big model in 64 bits."""
    g = np.random.default_rng(seed + 77)
    x = np.stack([system.x + 0.03 * g.standard_normal(system.x.shape) for _ in range(case["frames"])])
    ba = I.big_arch(system.n_species)
    ref = _Exact(system, ba, I.init_params(ba, SEED_BIG))
    e, f = [], []
    for k in range(len(x)):
        E, F = ref.energy_forces(torch.as_tensor(x[k], device="cuda"))
        e.append(E.sum())
        f.append(F)
    return torch.as_tensor(x, device="cuda"), torch.stack(f).contiguous(), torch.stack(e).contiguous()


def prepare(case, seed):
    system = _system(case, seed)
    sa, sp, ba, bp = _models(system.n_species)
    precision = D.BF16_MLP if case["precision"] == "bf16" else D.FP32
    opts = None
    if case.get("langevin"):
        opts = json.dumps({"langevin_friction": GAMMA_PS, "temperature": TEMPERATURE, "seed": seed % 100003})
    small = (None, None) if case.get("single") or case.get("model") == "big" else (sa, sp)
    ctx = D.Context(system, ba, bp, *small, precision=precision, options=opts)
    n = system.n_atoms
    st = {"case": case, "ctx": ctx}
    if case["kind"] == "distill":
        ctx.set_state(system.x)
        st["frames"], st["f_ref"], st["e_ref"] = _frames(case, system, seed)
        return st
    st["x"] = torch.as_tensor(system.x, device="cuda")
    st["f"] = torch.empty((n, 3), dtype=torch.float64, device="cuda")
    st["e"] = torch.empty(system.n_systems, dtype=torch.float64, device="cuda")
    if case["kind"] == "md":
        v = I.maxwell_boltzmann(system.mass, TEMPERATURE, seed + 1, system.atom_offset)
        st["v"] = torch.as_tensor(v, device="cuda")
        st["x_out"], st["v_out"] = torch.empty_like(st["x"]), torch.empty_like(st["x"])
    return st


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "forces":
        ctx.set_state(state["x"])
        which = D.BIG if case["model"] == "big" else D.SMALL
        out = ctx.forces(which, virial=case["virial"], f_out=state["f"], e_out=state["e"])
        got = {"energy": out[0].float(), "forces": out[1].float()}
        if case["virial"]:
            got["virial"] = out[2].astype(np.float32)
        return got
    if case["kind"] == "md":
        ctx.set_state(state["x"], state["v"])
        e = ctx.respa_step(case["n_outer"], case["dt"], case["n_inner"])
        x, v = ctx.get_state(state["x_out"], state["v_out"])
        return {"x": x.float(), "v": v.float(), "energies": e.astype(np.float32)}
    loss, grad = ctx.distill_grad(state["frames"], state["f_ref"], state["e_ref"], case["lambda_e"])
    return {"loss": np.float32(loss), "grad": grad.astype(np.float32)}


# ------------------------------------------------------------------ the same in 64 bits, by plain torch
class _Exact:
    """One potential in FP64: brute-force pairs, the energy written out, derivatives by torch."""

    def __init__(self, system, arch, params):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a, d=torch.float64: torch.as_tensor(np.asarray(a), dtype=d, device=self.dev)  # noqa: E731
        self.arch, self.n = arch, system.n_atoms
        self.theta = t(params)
        self.species = t(system.species, torch.int64)
        off = np.asarray(system.atom_offset)
        self.n_sys = len(off) - 1
        self.sid = t(np.repeat(np.arange(self.n_sys), np.diff(off)), torch.int64)
        self.lo, self.hi = t(off[:-1], torch.int64)[self.sid], t(off[1:], torch.int64)[self.sid]
        self.L = float(system.box[0])

    def pairs(self, x, cutoff):
        I_, J_ = [], []
        chunk = max(64, min(4096, (1 << 28) // max(1, self.n)))
        for a in range(0, self.n, chunk):
            b = min(self.n, a + chunk)
            c0, c1 = int(self.lo[a]), int(self.hi[b - 1])            # the systems these atoms belong to
            d2 = torch.zeros((b - a, c1 - c0), dtype=torch.float64, device=self.dev)
            for k in range(3):
                d = x[None, c0:c1, k] - x[a:b, None, k]
                if self.L > 0:
                    d -= self.L * torch.round(d / self.L)
                d2 += d * d
            keep = (d2 < cutoff * cutoff) & (self.sid[a:b, None] == self.sid[None, c0:c1])
            i = torch.arange(a, b, device=self.dev)
            keep[i - a, i - c0] = False
            p, q = torch.nonzero(keep, as_tuple=True)
            I_.append(p + a)
            J_.append(q + c0)
        return torch.cat(I_), torch.cat(J_)

    def blocks(self, theta):
        S, F, K = self.arch.n_species, self.arch.n_feat, self.arch.n_radial
        pos = 0

        def take(*shape):
            nonlocal pos
            m = math.prod(shape)
            pos += m
            return theta[pos - m:pos].reshape(shape)

        A = take(S, F)
        layers = [[take(F, F), take(K, F), take(F), take(F, F), take(F), take(F, F), take(F), take(F, F), take(F)]
                  for _ in range(self.arch.n_layers)]
        return A, layers, take(F, F), take(F), take(F), take(1), take(S)

    def energy(self, theta, i, j, r):
        a, silu = self.arch, torch.nn.functional.silu
        d = torch.sqrt((r * r).sum(1))
        k = torch.arange(1, a.n_radial + 1, dtype=torch.float64, device=self.dev)
        e = math.sqrt(2 / a.cutoff) * torch.sin(k * (math.pi / a.cutoff) * d[:, None]) / d[:, None]
        fc = 0.5 * (torch.cos(math.pi * d / a.cutoff) + 1)
        A, layers, R1, d1, R2, d2, e0 = self.blocks(theta)
        h = A[self.species]
        for W_in, W1, b1, W2, b2, U1, c1, U2, c2 in layers:
            w = fc[:, None] * (silu(e @ W1 + b1) @ W2 + b2)
            m = torch.zeros((self.n, a.n_feat), dtype=torch.float64, device=self.dev).index_add(0, i, w * (h @ W_in)[j])
            h = h + silu(m @ U1 + c1) @ U2 + c2
        E = silu(h @ R1 + d1) @ R2 + d2[0] + e0[self.species]
        on = d < a.rep_cutoff
        rep = 0.5 * a.rep_a * torch.exp(-d[on] / a.rep_rho) * 0.5 * (torch.cos(math.pi * d[on] / a.rep_cutoff) + 1)
        return E.index_add(0, i[on], rep)

    def per_system(self, E):
        return torch.zeros(self.n_sys, dtype=torch.float64, device=self.dev).index_add(0, self.sid, E)

    def geometry(self, x, pairs=None):
        i, j = self.pairs(x.detach(), self.arch.cutoff) if pairs is None else pairs
        r = x[j] - x[i]
        if self.L > 0:
            r = r - self.L * torch.round(r.detach() / self.L)
        return i, j, r

    def energy_forces(self, x, virial=False):
        """Per-system energies and forces; with virial also W = -sum over pairs of r (x) dE/dr."""
        i, j, r = self.geometry(x)
        r.requires_grad_(True)
        E = self.energy(self.theta, i, j, r)
        (g,) = torch.autograd.grad(E.sum(), r)
        f = torch.zeros((self.n, 3), dtype=torch.float64, device=self.dev).index_add(0, i, g).index_add(0, j, -g)
        out = (self.per_system(E.detach()), f)
        if virial:
            w = -(r.detach()[:, :, None] * g[:, None, :])
            out += (torch.zeros((self.n_sys, 3, 3), dtype=torch.float64, device=self.dev).index_add(0, self.sid[i], w),)
        return out

    def distill(self, frames, f_ref, e_ref, lambda_e):
        th = self.theta.clone().requires_grad_(True)
        loss_sum, grad = 0.0, torch.zeros_like(self.theta)
        for x, fr, er in zip(frames, f_ref, e_ref):
            i, j, r = self.geometry(x)
            r.requires_grad_(True)
            E = self.energy(th, i, j, r).sum()
            (g,) = torch.autograd.grad(E, r, create_graph=True)
            f = torch.zeros((self.n, 3), dtype=torch.float64, device=self.dev).index_add(0, i, g).index_add(0, j, -g)
            loss = (((f - fr) ** 2).sum() / (3 * self.n) + lambda_e * ((E - er) / self.n) ** 2) / len(frames)
            grad += torch.autograd.grad(loss, th)[0]
            loss_sum += float(loss.detach())
        return loss_sum, grad


def _philox_normals(n, step, seed, dev):
    """Three normals per atom: Philox-4x32-10 of counter (atom, step, 0, 0), key (seed, 0), Box-Muller."""
    M = 0xFFFFFFFF
    c = [torch.arange(n, dtype=torch.int64, device=dev), torch.full((n,), step, dtype=torch.int64, device=dev),
         torch.zeros(n, dtype=torch.int64, device=dev), torch.zeros(n, dtype=torch.int64, device=dev)]

    def mul(a, m):                      # 32 x 32 -> (high, low) words, through 16-bit halves
        lo, hi = (a & 0xFFFF) * m, (a >> 16) * m
        t = hi + (lo >> 16)
        return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)

    k0, k1 = seed & M, 0
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & M, (k1 + 0xBB67AE85) & M
    u = [(w.double() + 0.5) / 4294967296.0 for w in c]
    r01, r23 = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
    t = 2 * math.pi
    return torch.stack([r01 * torch.cos(t * u[1]), r01 * torch.sin(t * u[1]), r23 * torch.cos(t * u[3])], 1)


def _exact_md(case, seed, system):
    sa, sp, ba, bp = _models(system.n_species)
    big = _Exact(system, ba, bp)
    small = big if case["single"] else _Exact(system, sa, sp)
    dev, L = big.dev, big.L
    x = torch.as_tensor(system.x, device=dev)
    v = torch.as_tensor(I.maxwell_boltzmann(system.mass, TEMPERATURE, seed + 1, system.atom_offset), device=dev)
    m = torch.as_tensor(system.mass, device=dev)[:, None]
    wrap = (lambda y: y - L * torch.floor(y / L)) if L > 0 else (lambda y: y)
    n_in = case["n_inner"]
    h = case["dt"] / n_in
    x = wrap(x)
    c1 = math.exp(-GAMMA_PS * 1e-3 * h)
    sigma = math.sqrt(1 - c1 * c1) * torch.sqrt(KB_EV * TEMPERATURE * ACCEL / m)
    E, F = big.energy_forces(x)
    Fs = F if case["single"] else small.energy_forces(x)[1]
    step, out = 0, []
    for _ in range(case["n_outer"]):
        if not case["single"]:
            v = v + 0.5 * case["dt"] * ACCEL / m * (F - Fs)
        for k in range(n_in):
            v = v + 0.5 * h * ACCEL / m * Fs
            x = wrap(x + 0.5 * h * v)
            if case["langevin"]:
                v = c1 * v + sigma * _philox_normals(system.n_atoms, step, seed % 100003, dev)
            x = wrap(x + 0.5 * h * v)
            step += 1
            if case["single"]:
                E, F = big.energy_forces(x)
                Fs = F
            else:
                Fs = small.energy_forces(x)[1]
            v = v + 0.5 * h * ACCEL / m * Fs
        if not case["single"]:
            E, F = big.energy_forces(x)
            v = v + 0.5 * case["dt"] * ACCEL / m * (F - Fs)
        ke = big.per_system((0.5 * m[:, 0] * (v * v).sum(1)) / ACCEL)
        out.append(torch.stack([E, ke, E + ke], 1))
    return {"x": x, "v": v, "energies": torch.stack(out)}


def exact(case, seed):
    system = _system(case, seed)
    sa, sp, ba, bp = _models(system.n_species)
    if case["kind"] == "forces":
        arch, par = (ba, bp) if case["model"] == "big" else (sa, sp)
        ref = _Exact(system, arch, par)
        got = ref.energy_forces(torch.as_tensor(system.x, device=ref.dev), case["virial"])
        return dict(zip(("energy", "forces", "virial"), got))
    if case["kind"] == "md":
        return _exact_md(case, seed, system)
    loss, grad = _Exact(system, sa, sp).distill(*_frames(case, system, seed), case["lambda_e"])
    return {"loss": loss, "grad": grad}
