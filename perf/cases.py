"""What the engine is timed on: single passes through its public entry points.

A case names a molecule of ``qmc_inputs`` (with its bond length, its number of
determinants and whether it carries the many-body Jastrow), a precision form, a
number of walkers and a task:

* ``energy``    one ``Wavefunction.local_energy`` (E_L and log|Psi| per walker);
* ``sample``    ``Wavefunction.sample``: a stretch of a Metropolis chain that
                goes on from pass to pass, as between two optimisation steps;
* ``gradient``  one ``Wavefunction.energy_grad``: mean and variance of E_L, the
                parameter gradient and, where the entry point gives them, the
                forces on the nuclei.

Walkers.  A program evaluates energies and gradients on walkers of a Markov
chain, which follow |Psi|^2 and keep off its nodes; the start of a chain is a
Gaussian cloud round the nuclei.  ``prepare`` draws that cloud and, for the
energy and gradient tasks, takes a few Metropolis steps with the plain torch
wavefunction below (a walker near a node leaves it at the first move).

The torch code is written from the method's formulas in 64 bits and shares
nothing with the engine: it gives ``exact`` its values (E_L through analytic
orbital derivatives, or autograd Laplacians with backflow; gradients and forces
by autograd; chains with their own Philox4x32-10).
"""
import math

import numpy as np
import torch

import qmc_inputs as qi
from paper_2506_09743_gb300 import Wavefunction

DEV = "cuda"
F64 = torch.float64

# ---------------------------------------------------------------------------
# the cases


def _case(name, task, molecule, precision, walkers, **more):
    c = {"name": name, "task": task, "molecule": molecule, "precision": precision, "walkers": walkers,
         "bond": 1.0, "n_det": 1, "manybody": False}
    c.update(more)
    return c


def listed():
    return [
        # the smallest workload: a textbook molecule, where launches are the cost
        _case("h2_energy_fp64_1k", "energy", "h2", "fp64", 1024),
        # LiH at its workload size, headline form
        _case("lih_energy_fp32x2_64k", "energy", "lih", "fp32x2", 65536),
        # inverse backflow, a walker count that fills no tile
        _case("li2_energy_fp32x2_50k", "energy", "li2", "fp32x2", 50001),
        # a small ragged batch of the headline wavefunction: a short request
        _case("co_energy_fp32x2_4k", "energy", "co", "fp32x2", 4099, n_det=100),
        # the headline workload
        _case("co_energy_fp32x2_256k", "energy", "co", "fp32x2", 262144, n_det=100),
        # the fast form at a serving request's size
        _case("co_energy_tf32_64k", "energy", "co", "mixed_tf32", 65536, n_det=100),
        # the reference form: what optimisation and validation run
        _case("co_energy_fp64_16k", "energy", "co", "fp64", 16384, n_det=100),
        # the many-body Jastrow
        _case("co_mbj_energy_fp32x2_64k", "energy", "co", "fp32x2", 65536, n_det=100, manybody=True),
        # resampling between two optimisation steps: 10^4 walkers, the optimiser's form
        _case("lih_sample_fp64_10k", "sample", "lih", "fp64", 10000, steps=50, step=0.05),
        # a serving request's chain
        _case("co_sample_fp32x2_16k", "sample", "co", "fp32x2", 16384, n_det=100, steps=50, step=0.2),
        # an optimisation step's gradient with forces, backflow, 10^4 walkers
        _case("li2_gradient_fp64_10k", "gradient", "li2", "fp64", 10000),
        # the gradient of a determinant expansion (1,008 parameters)
        _case("co_gradient_fp64_64k", "gradient", "co", "fp64", 65536, n_det=100),
    ]


# (task, molecule, precision, most walkers): a drawn case costs no more than
# the largest listed one
_RANGES = (
    ("energy", "h2", "fp64", 262144), ("energy", "h2", "fp32x2", 262144),
    ("energy", "lih", "fp64", 262144), ("energy", "lih", "fp32x2", 262144), ("energy", "lih", "mixed_tf32", 262144),
    ("energy", "li2", "fp64", 131072), ("energy", "li2", "fp32x2", 262144),
    ("energy", "co", "fp64", 65536), ("energy", "co", "fp32x2", 262144), ("energy", "co", "mixed_tf32", 262144),
    ("sample", "h2", "fp64", 16384), ("sample", "lih", "fp64", 16384), ("sample", "lih", "fp32x2", 16384),
    ("sample", "li2", "fp64", 10000), ("sample", "co", "fp32x2", 16384), ("sample", "co", "mixed_tf32", 16384),
    ("gradient", "lih", "fp64", 32768), ("gradient", "li2", "fp64", 32768), ("gradient", "co", "fp64", 65536),
)


def draw(rng):
    task, molecule, precision, most = rng.choice(_RANGES)
    walkers = int(round(math.exp(rng.uniform(math.log(512), math.log(most)))))
    c = _case("", task, molecule, precision, walkers)
    del c["name"]
    c["bond"] = round(rng.uniform(0.6, 2.5), 2)  # the serving mix's stretch of the bond
    if molecule == "co":
        c["n_det"] = rng.choice((1, 20, 100))
        c["manybody"] = task == "energy" and precision != "fp64" and rng.random() < 0.25
    if task == "sample":
        c["steps"] = rng.choice((1, 5, 20, 50))
        c["step"] = rng.choice((0.05, 0.2))
    return c


def _molecule(case):
    kw = {"n_det": case["n_det"]} if case["molecule"] == "co" else {}
    mol = qi.make_molecule(case["molecule"], **kw).with_bond_scale(case["bond"])
    return qi.with_manybody_jastrow(mol) if case["manybody"] else mol


# ---------------------------------------------------------------------------
# the engine's side


def _start_walkers(case, seed, mol):
    """[3N, W] on the device: the Gaussian cloud a chain starts from."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) * 7919 + 17)
    home = torch.tensor(mol.atom_xyz[mol.electron_home], dtype=F64, device=DEV).reshape(-1, 1)
    z = torch.randn(3 * mol.n_elec, case["walkers"], dtype=F64, device=DEV, generator=g)
    return home + z, g


def _inputs(case, seed):
    """The molecule and the walkers [3N, W] of one state."""
    mol = _molecule(case)
    x, g = _start_walkers(case, seed, mol)
    if case["task"] != "sample":  # off the nodes, as a chain's walkers are
        psi = _Psi(mol)
        lp = _log_psi_soa(psi, x)
        for _ in range(4):
            y = x + 0.2 * torch.randn(x.shape, dtype=F64, device=DEV, generator=g)
            u = torch.rand(x.shape[1], dtype=F64, device=DEV, generator=g)
            lq = _log_psi_soa(psi, y)
            take = torch.log(u) < 2.0 * (lq - lp)
            x, lp = torch.where(take, y, x), torch.where(take, lq, lp)
    return mol, x.contiguous()


def prepare(case, seed):
    mol, x = _inputs(case, seed)
    s = {"case": case, "wf": Wavefunction(mol, precision=case["precision"]), "walkers": x, "seed": int(seed)}
    if case["task"] == "sample":
        s["log_psi"] = torch.empty(case["walkers"], dtype=F64, device=DEV)
        s["accepted"] = torch.zeros(case["walkers"], dtype=torch.int64, device=DEV)
        s["done"] = 0
    return s


def run(state):
    case, wf, x = state["case"], state["wf"], state["walkers"]
    if case["task"] == "energy":
        e, lp = wf.local_energy(x)
        return {"e_loc": e, "log_psi": lp}
    if case["task"] == "sample":
        wf.sample(x, case["steps"], case["step"], state["seed"], step_offset=state["done"],
                  log_psi=state["log_psi"], n_accept=state["accepted"])
        state["done"] += case["steps"]
        return {"walkers": x, "log_psi": state["log_psi"], "accepted": state["accepted"]}
    forces = case["molecule"] != "co"  # forces need a single determinant
    mean, var, grad, f = wf.energy_grad(x, want_forces=forces)
    out = {"mean": mean, "variance": var, "gradient": grad}
    if forces:
        out["forces"] = f
    return out


def work(case):
    """One pass: walkers read once, results written once; the formulas' flops
    (a primitive's exponential counted as one), every factor formed once."""
    mol = _molecule(case)
    n, na, W = mol.n_elec, mol.n_atom, case["walkers"]
    shells, prims = 0, 0
    key = None
    for b in range(mol.n_ao):  # AOs of one shell share their radial factor
        p0, p1 = int(mol.ao_prim_start[b]), int(mol.ao_prim_start[b + 1])
        k = (int(mol.ao_atom[b]), int(mol.ao_pow[b][:3].sum()), tuple(mol.prim_exp[p0:p1]))
        if k != key:
            shells, prims, key = shells + 1, prims + p1 - p0, k
    deriv = case["task"] != "sample"
    nch = 2 if deriv else 1
    if mol.backflow_w != 0.0 and deriv:
        nch = 10  # value, gradient and Hessian
    ncol = mol.n_mo if mol.n_det > 1 else max(mol.n_up, mol.n_down)
    ao = n * (8 * na + prims * (3 + 4 * (nch > 1)) + mol.n_ao * (2 * nch + 2 * nch * ncol))
    det = 0.0
    for m in (mol.n_up, mol.n_down):
        det += 2.0 * m ** 3 + (nch - 1) * 2.0 * m * m + (ncol - m) * nch * 2.0 * m * m
    det += 8.0 * mol.n_det
    if mol.backflow_w != 0.0 and deriv:
        det += 3 * n * (mol.n_up + mol.n_down) * (30.0 + 8.0 * max(mol.n_up, mol.n_down))
    pairs = n * (n - 1) / 2 * (40.0 if deriv else 20.0) + n * na * 10.0
    if case["manybody"]:
        pairs += n * (n - 1) / 2 * na * 5 * 30.0
    flops, in_out = ao + det + pairs, 24.0 * n
    if case["task"] == "energy":
        return {"bytes": W * (in_out + 16.0), "flops": W * flops}
    if case["task"] == "sample":  # the chain's steps build on one another: positions in, positions out
        return {"bytes": W * (2 * in_out + 24.0), "flops": W * case["steps"] * (flops + 30.0 * n)}
    n_param = int(mol.prim_exp.size) + mol.n_ao * mol.n_mo + mol.n_det + 2
    grad = n * (prims * 4 + mol.n_ao * (4.0 * ncol + 6))
    if case["molecule"] != "co":
        grad += 3.0 * na * flops  # a tangent of the whole energy per nuclear coordinate
    return {"bytes": W * in_out + 8.0 * n_param, "flops": W * (flops + grad)}


# ---------------------------------------------------------------------------
# the plain torch wavefunction (64 bits, on the device)


def _dfact(n):
    return 1.0 if n <= 1 else n * _dfact(n - 2)


class _Psi:
    """log|Psi| = J + log|sum_n d_n D_n^up D_n^down| of a molecule, with the
    parameters and the nuclei as tensors (``free`` makes them leaves)."""

    def __init__(self, mol, free=False):
        def t(a, dt=F64):
            return torch.tensor(np.asarray(a), dtype=dt, device=DEV)

        self.mol = mol
        # radial functions: one per run of AOs of a shell, or, where exponents
        # are differentiated, one per AO (each AO owns its primitives)
        P = max(int(mol.ao_prim_start[b + 1] - mol.ao_prim_start[b]) for b in range(mol.n_ao))
        keys, prim, shell_of = [], [], []
        for b in range(mol.n_ao):
            p0, p1 = int(mol.ao_prim_start[b]), int(mol.ao_prim_start[b + 1])
            ell, kn = int(mol.ao_pow[b][:3].sum()), int(mol.ao_pow[b][3])
            k = (int(mol.ao_atom[b]), int(mol.ao_kind[b]), ell, kn, tuple(mol.prim_exp[p0:p1]),
                 tuple(mol.prim_coef[p0:p1]), b if free else -1)
            if not keys or keys[-1] != k:
                keys.append(k)
                prim.append([p0 + q if q < p1 - p0 else -1 for q in range(P)])
            shell_of.append(len(keys) - 1)
        self.gto = bool(mol.ao_kind[0] == qi.GTO)
        assert all(int(k) == int(mol.ao_kind[0]) for k in mol.ao_kind)
        prim = np.asarray(prim)
        self.prim = t(np.maximum(prim, 0), torch.int64)
        self.prim_on = t(prim >= 0)
        self.shell_atom = t([k[0] for k in keys], torch.int64)
        self.ell, self.kn = t([k[2] for k in keys]), t([k[3] for k in keys])
        self.shell_of = t(shell_of, torch.int64)
        pw = np.asarray(mol.ao_pow)[:, :3]
        self.pw = t(pw, torch.int64)
        self.ao_atom = t(mol.ao_atom, torch.int64)
        df = np.array([_dfact(2 * a - 1) * _dfact(2 * b - 1) * _dfact(2 * c - 1) for a, b, c in pw])
        if self.gto:
            self.ang = t(1.0 / np.sqrt(df))
        else:
            self.ang = t([math.sqrt(_dfact(2 * int(p.sum()) + 1) / (4.0 * math.pi * d)) for p, d in zip(pw, df)])
        self.norm_sto = t([math.sqrt(math.factorial(2 * (k[2] + k[3] + 1))) for k in keys])
        self.R, self.Z = t(mol.atom_xyz), t(mol.atom_z)
        self.exps, self.coef, self.C = t(mol.prim_exp), t(mol.prim_coef), t(mol.mo_coeff)
        self.d, self.b, self.w = t(mol.det_weight), t(mol.jastrow_b), t(mol.backflow_w)
        self.jen = None if mol.jastrow_en is None else t(mol.jastrow_en)
        self.jeen = None if mol.jastrow_een is None else t(mol.jastrow_een)
        if free:
            for p in self.params() + [self.R]:
                p.requires_grad_(True)
        self.backflow = free or mol.backflow_w != 0.0
        up = torch.arange(mol.n_elec, device=DEV) < mol.n_up
        same = up[:, None] == up[None, :]
        i, j = torch.triu_indices(mol.n_elec, mol.n_elec, 1, device=DEV)
        self.i, self.j = i, j
        self.w0 = torch.where(same[i, j], float(mol.jastrow_w0_par), float(mol.jastrow_w0_anti)).to(F64)
        # excitations: flat offsets into T [n, n_mo] of the 2 x 2 block, per spin
        self.exc = []
        for s, n in ((0, mol.n_up), (1, mol.n_down)):
            e = np.asarray(mol.det_exc)[:, s, :]
            rank, h1, h2, p1, p2 = (e[:, k] for k in range(5))
            q = [np.where(rank >= r, h * mol.n_mo + p, 0) for r, h, p in
                 ((1, h1, p1), (2, h1, p2), (2, h2, p1), (2, h2, p2))]
            self.exc.append((n, t(rank, torch.int64), [t(v, torch.int64) for v in q]))

    def params(self):
        return [self.exps, self.C, self.d, self.b, self.w]

    def jastrow(self, r):
        v = r[:, self.i] - r[:, self.j]
        d = v.square().sum(-1).sqrt()
        J = (self.w0 * d / (1.0 + self.b * d)).sum(1)
        if self.jen is not None or self.jeen is not None:
            x = (r[:, :, None, :] - self.R).square().sum(-1).sqrt()  # [W, N, A]
        if self.jen is not None:
            w0, w1, w2 = self.jen
            J = J + ((w0 * x + w1 * x * x) / (1.0 + w2 * x)).sum((1, 2))
        if self.jeen is not None:
            def f(a, b, y):
                return a * y / (1.0 + b * y)

            for c, a1, b1, a2, b2, a3, b3 in self.jeen:
                f1, f2 = f(a1, b1, x), f(a2, b2, x)
                g = 0.5 * (f1[:, self.i] * f2[:, self.j] + f1[:, self.j] * f2[:, self.i]).sum(2)
                J = J + c * (g * f(a3, b3, d)).sum(1)
        return J

    def potential(self, r):
        d = (r[:, self.i] - r[:, self.j]).square().sum(-1).sqrt()
        x = (r[:, :, None, :] - self.R).square().sum(-1).sqrt()
        V = (1.0 / d).sum(1) - (self.Z / x).sum((1, 2))
        for a in range(self.mol.n_atom):
            for b in range(a + 1, self.mol.n_atom):
                V = V + self.Z[a] * self.Z[b] / (self.R[a] - self.R[b]).square().sum().sqrt()
        return V

    def positions(self, r):
        """r~_i = r_i + sum_j (w / r_ij)(r_i - r_j)."""
        if not self.backflow:
            return r
        v = r[:, self.i] - r[:, self.j]
        g = v / v.square().sum(-1, keepdim=True).sqrt()
        z = torch.zeros_like(r)
        return r + self.w * (z.index_add(1, self.i, g) - z.index_add(1, self.j, g))

    def orbitals(self, q, derivs=False):
        """MO values at q [W, N, 3]; with derivs also gradients and Laplacians."""
        dv = q[:, :, None, :] - self.R  # [W, N, A, 3]
        r2 = dv.square().sum(-1)
        r2s = r2[..., self.shell_atom]
        a = self.exps[self.prim]
        c = self.coef[self.prim] * self.prim_on
        if self.gto:
            c = c * (2.0 * a / math.pi) ** 0.75 * (4.0 * a) ** (0.5 * self.ell[:, None])
            e = c * torch.exp(-a * r2s[..., None])
            f = e.sum(-1)
            if derivs:
                t1 = (2.0 * a * e).sum(-1)
                g1, f2 = -t1, r2s * (4.0 * a * a * e).sum(-1) - t1
        else:
            a, c = a[:, 0], c[:, 0]
            rho = r2s.sqrt()
            n = self.kn + self.ell + 1.0
            f = c * (2.0 * a) ** (n + 0.5) / self.norm_sto * torch.exp(-a * rho)
            f = f * torch.where(self.kn > 0, rho ** self.kn, torch.ones_like(rho))
            if derivs:
                h = self.kn / rho - a
                g1, f2 = h * f / rho, (h * h - self.kn / r2s) * f
        top = int(self.pw.max()) + 1
        pows = torch.stack([torch.ones_like(dv)] + [dv ** k for k in range(1, top)], -1)  # [W, N, A, 3, K]

        def mono(k):  # x^kx y^ky z^kz of every AO, k [n_ao, 3]; negative powers give 0
            on = (k >= 0).all(1)
            k = k.clamp_min(0)
            P = pows[:, :, self.ao_atom, 0, k[:, 0]] * pows[:, :, self.ao_atom, 1, k[:, 1]]
            return P * pows[:, :, self.ao_atom, 2, k[:, 2]] * on

        P, fa = mono(self.pw), f[..., self.shell_of]
        M = self.ang[:, None] * self.C
        phi = (P * fa) @ M
        if not derivs:
            return phi
        one = torch.eye(3, dtype=torch.int64, device=DEV)
        g1a, grad, lap = g1[..., self.shell_of], [], 0.0
        for k in range(3):
            dP = self.pw[:, k] * mono(self.pw - one[k])
            grad.append((fa * dP + P * g1a * dv[:, :, self.ao_atom, k]) @ M)
            lap = lap + self.pw[:, k] * (self.pw[:, k] - 1) * mono(self.pw - 2 * one[k])
        rad = (f2 + 2.0 * (self.ell + 1.0) * g1)[..., self.shell_of]
        return phi, grad, (fa * lap + P * rad) @ M

    def log_sum(self, phi):
        """log|sum_n d_n D_n^up D_n^down| from the MO values [W, N, n_mo]."""
        out, ratio, i0 = 0.0, [], 0
        for n, rank, (q00, q01, q10, q11) in self.exc:
            W = phi.shape[0]
            if n == 0:
                ratio.append(torch.ones(W, len(rank), dtype=F64, device=DEV))
                continue
            rows = phi[:, i0:i0 + n]
            A = rows[:, :, :n]
            out = out + torch.linalg.slogdet(A)[1]
            if int(rank.max()) == 0:
                ratio.append(torch.ones(W, len(rank), dtype=F64, device=DEV))
            else:
                T = (torch.linalg.inv(A) @ rows).reshape(W, -1)
                s00 = T[:, q00]
                R = torch.where(rank == 0, torch.ones_like(s00), s00)
                if int(rank.max()) == 2:
                    R = torch.where(rank == 2, s00 * T[:, q11] - T[:, q01] * T[:, q10], R)
                ratio.append(R)
            i0 += n
        return out + ((ratio[0] * ratio[1]) @ self.d).abs().log()

    def log_psi(self, r):
        return self.jastrow(r) + self.log_sum(self.orbitals(self.positions(r)))

    def energy(self, r, graph=False):
        """(E_L, log|Psi|); with graph the energy can be differentiated again."""
        r = r.detach().requires_grad_(True)
        if self.backflow:
            lp = self.log_psi(r)
            g, lap = _grad_lap(lp, r, graph)
            return -0.5 * (lap + g.square().sum((1, 2))) + self.potential(r), lp
        J = self.jastrow(r)
        g, lap = _grad_lap(J, r, False)
        with torch.no_grad():
            phi, dphi, kin = self.orbitals(r, True)
            for k in range(3):
                kin = kin + 2.0 * g[:, :, k, None] * dphi[k]
        phi.requires_grad_(True)
        ls = self.log_sum(phi)
        # the kinetic operator moves the orbitals along kin: its trace over the
        # expansion is the derivative of log|Sigma| in that direction
        slater = (torch.autograd.grad(ls.sum(), phi)[0] * kin).sum((1, 2))
        e = -0.5 * (lap + g.square().sum((1, 2)) + slater) + self.potential(r)
        return e.detach(), (J + ls).detach()


def _grad_lap(y, r, graph):
    """Gradient and Laplacian of y [W] with respect to r [W, N, 3]."""
    g = torch.autograd.grad(y.sum(), r, create_graph=True)[0]
    lap = 0.0
    for i in range(r.shape[1]):
        for k in range(3):
            h = torch.autograd.grad(g[:, i, k].sum(), r, create_graph=graph, retain_graph=True)[0]
            lap = lap + h[:, i, k]
    return (g if graph else g.detach()), lap


def _electrons(x):
    """[3N, W] -> [W, N, 3]."""
    return x.t().reshape(x.shape[1], -1, 3)


def _log_psi_soa(psi, x, chunk=32768):
    with torch.no_grad():
        return torch.cat([psi.log_psi(_electrons(x[:, k:k + chunk])) for k in range(0, x.shape[1], chunk)])


def _philox(seed, j, walker, step):
    """Philox4x32-10 words of counter (j, walker, step) under key seed."""
    mask = 0xFFFFFFFF

    def mul(a, x):  # high and low words of a x
        lo, hi = a * (x & 0xFFFF), a * (x >> 16)
        mid = hi + (lo >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    c = [torch.full_like(walker, j), walker & mask, torch.full_like(walker, step & mask),
         torch.full_like(walker, step >> 32)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for q in range(10):
        if q:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    return [(v.to(F64) + 0.5) * 2.0 ** -32 for v in c]


def _exact_chain(case, seed, psi, x):
    """The Metropolis chain of Gaussian moves of all electrons at once."""
    n3, W = x.shape
    walker = torch.arange(W, dtype=torch.int64, device=DEV)
    lp = _log_psi_soa(psi, x)
    blocks = (n3 + 3) // 4
    for step in range(case["steps"]):
        z = []
        for j in range(blocks):
            u = _philox(int(seed), j, walker, step)
            for a, b in ((0, 1), (2, 3)):
                rad = (-2.0 * torch.log(u[a])).sqrt()
                z += [rad * torch.cos(2.0 * math.pi * u[b]), rad * torch.sin(2.0 * math.pi * u[b])]
        y = x + case["step"] * torch.stack(z[:n3])
        lq = _log_psi_soa(psi, y)
        take = torch.log(_philox(int(seed), blocks, walker, step)[0]) < 2.0 * (lq - lp)
        x, lp = torch.where(take, y, x), torch.where(take, lq, lp)
    return {"walkers": x, "log_psi": lp, "accepted": None}


def exact(case, seed):
    mol, x = _inputs(case, seed)
    W = x.shape[1]
    if case["task"] == "sample":
        # the lower-precision forms decide a few acceptances otherwise: their
        # chains have no 64-bit value
        return _exact_chain(case, seed, _Psi(mol), x) if case["precision"] == "fp64" else None
    if case["task"] == "energy":
        psi, e, lp = _Psi(mol), [], []
        for k in range(0, W, 16384):
            a, b = psi.energy(_electrons(x[:, k:k + 16384]))
            e.append(a.detach())
            lp.append(b.detach())
        return {"e_loc": torch.cat(e), "log_psi": torch.cat(lp)}
    # gradient: 2 <(E - <E>) d log|Psi|>, forces -<dE/dR + (E - <E>) d ln|Psi|^2/dR>
    forces = case["molecule"] != "co"
    plain, e, chunk = _Psi(mol), [], 4096
    for k in range(0, W, chunk):
        e.append(plain.energy(_electrons(x[:, k:k + chunk]))[0].detach())
    e = torch.cat(e)
    mean, dev = e.mean(), e - e.mean()
    psi = _Psi(mol, free=True)
    grad, f = None, torch.zeros_like(psi.R)
    for k in range(0, W, chunk):
        r = _electrons(x[:, k:k + chunk])
        lp = psi.log_psi(r)
        need = psi.params() + [psi.R]
        g = torch.autograd.grad((2.0 / W * dev[k:k + chunk] * lp).sum(), need)
        grad = list(g[:-1]) if grad is None else [a + b for a, b in zip(grad, g[:-1])]
        if forces:
            el, _ = psi.energy(r, graph=True)
            f = f - g[-1] - torch.autograd.grad(el.sum() / W, psi.R)[0]
            del el
    out = {"mean": mean, "variance": dev.square().mean(), "gradient": torch.cat([g.reshape(-1) for g in grad])}
    if forces:
        out["forces"] = f
    return out
