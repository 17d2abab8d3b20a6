"""GPU parity of the stages that serve one kind of wavefunction, at the edges
of what they take: ragged warps and tiles, the smallest and largest electron
counts, shells in any order, incomplete or of higher angular momentum, many
parameters.

Tolerances, fixed before measurement: energies as in gpu_common; the two forms
of the tensor-core FP32X2 AO stage bit for bit (every product and sum behind
the digits is exact, so they may not differ); gradients at 1e-8 of the largest
component, the criterion of the workloads' gradient tests; the mean at 1e-10
of the largest energy and the variance at 1e-8 of itself or of 1e-10 times the
largest energy squared, the energies being within 1e-11 or so of each other.
"""
import dataclasses

import numpy as np
import pytest
import torch

import qmc_inputs as qi
from gpu_common import fp32ao_check, fp64_check, gated_check, oracle_reference
from oracle import qmc_oracle as O

pytestmark = pytest.mark.gpu

F_SHELL = [(3, 0, 0), (0, 3, 0), (0, 0, 3), (2, 1, 0), (2, 0, 1), (1, 2, 0), (0, 2, 1), (1, 0, 2), (0, 1, 2), (1, 1, 1)]


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    import paper_2506_09743_gb300 as p

    return p


def _mol(n_up, n_down, shells, n_mo, n_det=1, n_prim=3, sto=False, seed=0):
    """Three nuclei with the given shells each ("s", "p", "d", "f": complete, the
    functions in another order every time; "P", "D": one function left out),
    random orbitals, a leading determinant and random excitations."""
    rng = np.random.default_rng(1000 * n_up + 100 * n_down + 10 * n_mo + n_det + seed)
    bb = qi._BasisBuilder()
    parts = {"s": [(0, 0, 0)], "p": qi.P_SHELL, "d": qi.D_SHELL, "f": F_SHELL, "P": qi.P_SHELL[1:], "D": qi.D_SHELL[1:]}
    for a in range(3):
        for sh in shells:
            if sto:
                ex, co, kn = [rng.uniform(0.7, 2.0)], [1.0], int(rng.integers(2))
            else:
                ex, co, kn = rng.uniform(0.2, 4.0, n_prim), rng.uniform(0.2, 1.0, n_prim), 0
            fns = parts[sh]
            for k in rng.permutation(len(fns)):
                bb.add(a, qi.STO if sto else qi.GTO, *fns[k], kn, ex, co)
    arr = bb.arrays()
    g = qi.ground_exc()
    dets = qi._select_dets(qi.sd_expansion(n_up, n_down, n_mo), n_det, rng) if n_det > 1 else [(g, g)]
    xyz = np.array([[0.0, 0.0, -1.2], [0.3, 0.2, 1.0], [1.3, -0.7, 0.1]])
    n = n_up + n_down
    w = rng.uniform(-0.1, 0.1, len(dets))
    w[0] = 0.9
    return qi.Molecule(name=f"e{n_up}.{n_down}.{shells}.{n_mo}.{n_det}.{n_prim}.{sto}.{seed}", atom_xyz=xyz,
                       atom_z=np.array([3.0, 2.0, max(1.0, n - 5.0)]), n_up=n_up, n_down=n_down, **arr,
                       mo_coeff=qi.random_orthonormal(len(arr["ao_atom"]), n_mo, rng), det_weight=w,
                       det_exc=qi._dets_array(dets), jastrow_b=0.9, electron_home=np.arange(n, dtype=np.int32) % 3)


def _x(r, pad=0):
    return torch.tensor(qi.to_soa(r, ldw=r.shape[0] + pad), device="cuda")


# -- FP64 AO stage: closed forms of complete shells, the general form of the rest
@pytest.mark.parametrize("shells", ["sspd", "sPd", "spD", "spdf", "dps"])
@pytest.mark.parametrize("n_mo,n_det", [(5, 1), (9, 4)])
@pytest.mark.parametrize("sto", [False, True])
def test_fp64_rows_of_any_shell(pkg, shells, n_mo, n_det, sto):
    mol = _mol(5, 4, shells, n_mo, n_det, sto=sto)
    r = qi.walkers(mol, 37, seed=3)
    E, lp, sens = oracle_reference(mol, r)
    wf = pkg.Wavefunction(mol)
    for W in (1, 37):
        e, _ = wf.local_energy(_x(r, 3), n_walkers=W)
        torch.cuda.synchronize()
        fp64_check(e.cpu().numpy(), E[:W], sens[:W], min_within=0.0)
    wf.close()


# -- one determinant, up to four orbitals per spin: one thread per walker
@pytest.mark.parametrize("n_up,n_down", [(2, 1), (2, 2), (3, 2), (3, 3), (4, 1), (4, 4), (3, 0)])
@pytest.mark.parametrize("precision", ["fp64", "fp32x2"])
def test_one_determinant_of_few_orbitals(pkg, n_up, n_down, precision):
    mol = _mol(n_up, n_down, "spd", max(n_up, n_down) + 2)
    r = qi.walkers(mol, 129, seed=4)
    E, lp, sens = oracle_reference(mol, r)
    # a 1 x 1 reference matrix has condition number one even where its orbital
    # vanishes: there the orbital's own cancellation counts
    owf = O.Wavefunction(mol)
    ao = O.ao_eval(owf, torch.tensor(r))
    for i, n in ((0, n_up), (n_up, n_down)):
        if n == 1:
            t = ao[:, i] * owf.mo[:, 0]
            sens = np.maximum(sens, (t.abs().sum(-1) / t.sum(-1).abs()).numpy())
    wf = pkg.Wavefunction(mol, precision=precision)
    for W in (1, 127, 129):
        e, _ = wf.local_energy(_x(r, 1), n_walkers=W)
        torch.cuda.synchronize()
        if precision == "fp64":
            fp64_check(e.cpu().numpy(), E[:W], sens[:W], min_within=0.0)
        else:
            gated_check(e.cpu().numpy(), E[:W], sens[:W])
    wf.close()


# -- FP32X2 Jastrow stage: walkers over lanes, pairs over warps
@pytest.mark.parametrize("n_up,n_down", [(4, 3), (7, 0), (5, 4), (7, 7), (8, 8)])
@pytest.mark.parametrize("mb", [False, True])
def test_wide_jastrow(pkg, n_up, n_down, mb):
    mol = _mol(n_up, n_down, "sspp", max(n_up, n_down) + 1)
    if mb:
        mol = dataclasses.replace(qi.with_manybody_jastrow(mol), name=mol.name + "mb")
    r = qi.walkers(mol, 33, seed=5)
    r[0, 1] = r[0, 0] + [0.03, -0.04, 0.0]  # a close pair
    r[31, 0] = mol.atom_xyz[2] + [0.0, 0.02, 0.01]  # an electron close to a nucleus
    E, lp, sens = oracle_reference(mol, r)
    wf = pkg.Wavefunction(mol, precision="fp32x2")
    for W in (1, 31, 32, 33):
        e, l = wf.local_energy(_x(r, 2), n_walkers=W)
        torch.cuda.synchronize()
        gated_check(e.cpu().numpy(), E[:W], sens[:W])
        keep = sens[:W] < 1e6
        assert np.all(np.abs(l.cpu().numpy() - lp[:W])[keep] <= 1e-5)
    wf.close()


# -- tensor-core FP32X2 AO stage: two rows per thread against one row per thread
@pytest.mark.parametrize("shells,n_mo", [("sssppd", 14), ("ddpss", 9), ("sppd", 16), ("ssssppp", 11)])
def test_packed_rows_match_single_rows(pkg, shells, n_mo):
    """A Slater function that no orbital contains, and that is far below every
    row's scale, takes the wavefunction to the one-row kernel and leaves every
    digit as it is."""
    mol = _mol(7, 6, shells, n_mo, 3, sto=False)
    plus = dataclasses.replace(
        mol, name=mol.name + "+", ao_atom=np.append(mol.ao_atom, np.int32(2)),
        ao_kind=np.append(mol.ao_kind, np.int32(qi.STO)), ao_pow=np.vstack([mol.ao_pow, [[0, 0, 0, 0]]]).astype(np.int32),
        ao_prim_start=np.append(mol.ao_prim_start, np.int32(mol.ao_prim_start[-1] + 1)),
        prim_exp=np.append(mol.prim_exp, 40.0), prim_coef=np.append(mol.prim_coef, 1e-30),
        mo_coeff=np.vstack([mol.mo_coeff, np.zeros((1, n_mo))]))
    r = qi.walkers(mol, 259, seed=6)
    r[2, 3] = mol.atom_xyz[1] + 1e-5  # on a nucleus, as far as the scales are concerned
    r[128, 0] = mol.atom_xyz[0] + [0.0, 1e-4, 0.0]
    r[64, 1] = [40.0, 3.0, 0.0]  # every AO tiny
    a, b = pkg.Wavefunction(mol, precision="fp32x2"), pkg.Wavefunction(plus, precision="fp32x2")
    for W in (1, 63, 64, 65, 127, 128, 129, 259):
        ea, la = a.local_energy(_x(r, 1), n_walkers=W)
        eb, lb = b.local_energy(_x(r, 1), n_walkers=W)
        torch.cuda.synchronize()
        assert torch.equal(torch.nan_to_num(ea), torch.nan_to_num(eb))
        assert torch.equal(torch.nan_to_num(la), torch.nan_to_num(lb))
        assert torch.isfinite(la).sum() >= W - 2
    a.close()
    b.close()


# -- TF32 AO stage: two rows per thread, shells of every kind
@pytest.mark.parametrize("shells", ["ssp", "sspd", "sPDf"])
@pytest.mark.parametrize("sto", [False, True])
def test_tf32_rows_of_any_shell(pkg, shells, sto):
    mol = _mol(5, 4, shells, 6, 3, sto=sto)
    r = qi.walkers(mol, 259, seed=9)
    E, lp, sens = oracle_reference(mol, r)
    wf = pkg.Wavefunction(mol, precision="mixed_tf32")
    full = None
    for W in (259, 129, 128, 65, 64, 63, 1):
        e, l = wf.local_energy(_x(r, 1), n_walkers=W)
        torch.cuda.synchronize()
        fp32ao_check(e.cpu().numpy(), E[:W], sens[:W])
        full = (e, l) if full is None else full
        assert torch.equal(e, full[0][:W]) and torch.equal(l, full[1][:W])  # a row does not depend on the batch
    # the value path (a chain of no steps returns log|Psi| of where it stands)
    x, lps = _x(r, 1), torch.empty(259, dtype=torch.float64, device="cuda")
    wf.sample(x, 0, 0.3, 5, n_walkers=259, log_psi=lps)
    torch.cuda.synchronize()
    assert np.all(np.abs(lps.cpu().numpy() - lp) <= 128 * 2.0 ** -24 * sens * np.maximum(1.0, np.abs(lp)))
    wf.close()


# -- gradient rows: tiles of 32 walkers, chunks of AOs and radial derivatives
@pytest.mark.parametrize("shells,n_mo,n_prim,sto", [("spd", 5, 3, False), ("sPDf", 7, 8, False), ("f", 4, 1, False),
                                                    ("spPd", 5, 1, True), ("s" * 6 + "p" * 6 + "d" * 10, 16, 8, False)])
@pytest.mark.parametrize("W", [2, 31, 33, 65])
def test_gradient_rows(pkg, shells, n_mo, n_prim, sto, W):
    """The last basis has 6,000 parameters: fewer warps per block."""
    mol = _mol(4, 3, shells, n_mo, 3 if n_mo > 4 else 1, n_prim=n_prim, sto=sto)
    if n_mo == 4:
        mol = qi.with_manybody_jastrow(mol)
    r = qi.walkers(mol, W, seed=7)
    _, _, g_ref, _ = O.energy_grad(O.Wavefunction(mol, requires_grad=True), torch.tensor(r))
    g_ref = g_ref.numpy()
    wf = pkg.Wavefunction(mol)
    _, _, g, _ = wf.energy_grad(_x(r, 5), n_walkers=W, want_forces=False)
    assert np.abs(g.cpu().numpy() - g_ref).max() <= 1e-8 * np.abs(g_ref).max()
    wf.close()


# -- mean and variance: chunks of 2,048 energies
@pytest.mark.parametrize("W", [1, 2, 2047, 2048, 2049, 4097, 40960])
def test_mean_and_variance_around_the_chunks(pkg, W):
    mol = qi.make_h2()
    x = _x(qi.walkers(mol, W, seed=8), 1)
    wf = pkg.Wavefunction(mol)
    e = wf.local_energy(x, n_walkers=W)[0].cpu().numpy()
    m, v, _, _ = wf.energy_grad(x, n_walkers=W, want_grad=False, want_forces=False)
    top = np.abs(e).max()
    assert abs(m - e.mean()) <= 1e-10 * top
    assert abs(v - e.var()) <= 1e-8 * e.var() + 1e-10 * top * top
    wf.close()


# -- small molecules: p functions held by shells of their own (as after an optimisation step)
@pytest.mark.parametrize("n_up,n_down", [(1, 1), (3, 2), (4, 4)])
@pytest.mark.parametrize("sto", [False, True])
@pytest.mark.parametrize("precision,w", [("fp64", 0.0), ("fp64", 0.1), ("fp32x2", 0.1)])
def test_split_p_shells_match_whole_ones(pkg, n_up, n_down, sto, precision, w):
    """The functions of two p shells of a nucleus written alternately (x, x, y,
    y, z, z) are six shells of one function: every sum keeps its order, so
    energies, log|Psi|, chains and parameter gradients are the same bit for bit.
    (The forces add the functions' terms in another order: 1e-12 of the largest.)"""
    mol = dataclasses.replace(_mol(n_up, n_down, "spp", max(n_up, n_down) + 1, n_prim=2, sto=sto), backflow_w=w)
    xyz = [int(np.argmax(k[:3])) for k in mol.ao_pow]  # axis of a p function
    order = []
    for a in range(3):  # per nucleus: s, then two p shells in any order
        b = 7 * a
        sh = [sorted(range(b + 1, b + 4), key=lambda k: xyz[k]), sorted(range(b + 4, b + 7), key=lambda k: xyz[k])]
        order.append([b] + sh[0] + sh[1])
    def pick(idx):
        n = np.diff(mol.ao_prim_start)
        pr = np.concatenate([np.arange(mol.ao_prim_start[k], mol.ao_prim_start[k + 1]) for k in idx])
        return dataclasses.replace(
            mol, ao_atom=mol.ao_atom[idx], ao_kind=mol.ao_kind[idx], ao_pow=mol.ao_pow[idx],
            ao_prim_start=np.concatenate([[0], np.cumsum(n[idx])]).astype(np.int32), prim_exp=mol.prim_exp[pr],
            prim_coef=mol.prim_coef[pr], mo_coeff=mol.mo_coeff[idx]), pr
    whole, pr_w = pick(np.concatenate(order))
    split, pr_s = pick(np.concatenate([[o[0], o[1], o[4], o[2], o[5], o[3], o[6]] for o in order]))
    x = _x(qi.walkers(mol, 45, seed=12), 2)
    a, b = pkg.Wavefunction(whole, precision=precision), pkg.Wavefunction(split, precision=precision)
    ea, la = a.local_energy(x, n_walkers=45)
    eb, lb = b.local_energy(x, n_walkers=45)
    torch.cuda.synchronize()
    assert torch.equal(ea, eb) and torch.equal(la, lb)
    ya, yb = x.clone(), x.clone()
    a.sample(ya, 5, 0.3, 13, n_walkers=45)
    b.sample(yb, 5, 0.3, 13, n_walkers=45)
    torch.cuda.synchronize()
    assert torch.equal(ya, yb)
    if precision == "fp64":
        _, _, ga, fa = a.energy_grad(x, n_walkers=45)
        _, _, gb, fb = b.energy_grad(x, n_walkers=45)
        ga, gb = ga.cpu().numpy(), gb.cpu().numpy()
        n = mol.prim_exp.size
        ta, tb = np.empty(n), np.empty(n)
        ta[pr_w], tb[pr_s] = ga[:n], gb[:n]
        assert np.array_equal(ta, tb)
        m = mol.mo_coeff.size
        ca, cb = np.empty(mol.mo_coeff.shape), np.empty(mol.mo_coeff.shape)
        ca[np.concatenate(order)] = ga[n:n + m].reshape(ca.shape)
        cb[np.concatenate([[o[0], o[1], o[4], o[2], o[5], o[3], o[6]] for o in order])] = gb[n:n + m].reshape(cb.shape)
        assert np.array_equal(ca, cb)
        assert np.abs((fa - fb).cpu().numpy()).max() <= 1e-12 * max(1.0, float(fa.abs().max()))
    a.close()
    b.close()
