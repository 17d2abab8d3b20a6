"""GPU parity of the small-molecule kernels (one lane per electron) at their
edges: every electron count and spin split they serve, empty spins, batches
that leave the last warp part full, Slater and Gaussian shells, p shells in an
order of their own, with and without backflow.

Tolerances as in gpu_common (fixed before measurement): energies by
fp64_check, log|Psi| within the same backward-error bound, FP32X2 by the
2e-4 Ha gate; the gradient and forces at 1e-8 of their largest component, the
criterion of the workloads' gradient tests.  A spin with a single electron has
a 1 x 1 reference matrix, whose condition number is one even where its orbital
vanishes: there the sensitivity takes the orbital's own cancellation,
sum_b |C_b phi_b| / |sum_b C_b phi_b|, in its place.
"""
import numpy as np
import pytest
import torch

import qmc_inputs as qi
from gpu_common import C_BOUND, U64, fp64_check, gated_check, oracle_reference
from oracle import qmc_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g

    g.build()
    import paper_2506_09743_gb300 as p

    return p


def _mol(n_up, n_down, gto, w):
    """Three nuclei, two s shells and one p shell each, random orbitals; the p
    functions of each shell in another order."""
    rng = np.random.default_rng(100 * n_up + 10 * n_down + gto)
    bb = qi._BasisBuilder()
    for a in range(3):
        for l_of in (0, 0, 1):
            if gto:
                ex, co, kn = rng.uniform(0.2, 3.0, 2), rng.uniform(0.2, 1.0, 2), 0
            else:
                ex, co, kn = [rng.uniform(0.5, 2.0)], [1.0], int(rng.integers(2))
            for p in ([(0, 0, 0)] if l_of == 0 else [qi.P_SHELL[k] for k in np.roll(range(3), a)]):
                bb.add(a, qi.GTO if gto else qi.STO, *p, kn, ex, co)
    n = n_up + n_down
    xyz = np.array([[0.0, 0.0, -1.1], [0.3, 0.2, 1.0], [1.2, -0.7, 0.1]])
    z = np.array([2.0, 1.0, float(max(1, n - 3))])
    n_mo = max(n_up, n_down) + 1
    mo = qi.random_orthonormal(15, n_mo, rng)
    g = qi.ground_exc()
    return qi.Molecule(name=f"s{n_up}{n_down}{gto}{w}", atom_xyz=xyz, atom_z=z, n_up=n_up, n_down=n_down, **bb.arrays(),
                       mo_coeff=mo, det_weight=np.array([0.8]), det_exc=qi._dets_array([(g, g)]), jastrow_b=0.9,
                       backflow_w=w, electron_home=np.arange(n, dtype=np.int32) % 3)


def _sensitivity(mol, r, sens):
    """The oracle's sensitivity, with the orbitals of single-electron spins."""
    wf = O.Wavefunction(mol)
    rt = torch.tensor(r)
    ao = O.ao_eval(wf, O.backflow(wf, rt) if wf.has_backflow else rt)  # [W, N, n_ao]
    for i, n in ((0, mol.n_up), (mol.n_up, mol.n_down)):
        if n == 1:
            t = ao[:, i] * wf.mo[:, 0]
            sens = np.maximum(sens, (t.abs().sum(-1) / t.sum(-1).abs()).numpy())
    return sens


SPINS = [(1, 0), (1, 1), (2, 1), (2, 2), (3, 0), (3, 2), (3, 3), (4, 1), (4, 3), (4, 4)]


@pytest.mark.parametrize("n_up,n_down", SPINS)
@pytest.mark.parametrize("gto", [0, 1])
@pytest.mark.parametrize("w", [0.0, 0.1])
def test_energy_gradient_and_chain_at_the_edges(pkg, n_up, n_down, gto, w):
    mol = _mol(n_up, n_down, gto, w)
    N = n_up + n_down
    per = 32 // N  # walkers per warp
    W = 3 * per + max(1, per // 2)
    r = qi.walkers(mol, W, seed=5)
    E, lp, sens = oracle_reference(mol, r)
    sens = _sensitivity(mol, r, sens)
    x = torch.tensor(qi.to_soa(r, ldw=W + 3), device="cuda")
    wf = pkg.Wavefunction(mol)
    for k in sorted({1, max(1, per - 1), per, min(W, per + 1), W}):
        e, l = wf.local_energy(x, n_walkers=k)
        torch.cuda.synchronize()
        fp64_check(e.cpu().numpy(), E[:k], sens[:k], min_within=0.0)
        bound = C_BOUND * U64 * sens[:k] * np.maximum(1.0, np.abs(lp[:k]))
        assert np.all(np.abs(l.cpu().numpy() - lp[:k]) <= bound)
    ev, var, g_ref, f_ref = O.energy_grad(O.Wavefunction(mol, requires_grad=True), torch.tensor(r))
    _, _, g, f = wf.energy_grad(x, n_walkers=W)
    g_ref, f_ref = g_ref.numpy(), f_ref.numpy()
    assert np.abs(g.cpu().numpy() - g_ref).max() <= 1e-8 * np.abs(g_ref).max()
    assert np.abs(f.cpu().numpy() - f_ref).max() <= 1e-8 * max(1.0, np.abs(f_ref).max())
    r_ref, lp_ref, acc_ref = O.metropolis(O.Wavefunction(mol), torch.tensor(r), 6, 0.3, seed=11)
    acc = torch.zeros(W, dtype=torch.int64, device="cuda")
    lps = torch.empty(W, dtype=torch.float64, device="cuda")
    wf.sample(x, 6, 0.3, 11, n_walkers=W, log_psi=lps, n_accept=acc)
    torch.cuda.synchronize()
    assert np.array_equal(acc.cpu().numpy(), acc_ref.numpy())
    assert np.abs(qi.from_soa(x.cpu().numpy(), W, N) - r_ref.numpy()).max() < 1e-10
    assert np.abs(lps.cpu().numpy() - lp_ref.numpy()).max() < 1e-9
    wf.close()


@pytest.mark.parametrize("n_up,n_down", [(1, 1), (2, 1), (3, 3), (4, 3), (4, 4)])
@pytest.mark.parametrize("gto", [0, 1])
def test_pair_orbitals_at_the_edges(pkg, n_up, n_down, gto):
    mol = _mol(n_up, n_down, gto, 0.1)
    W = 2 * (32 // (n_up + n_down)) + 1
    r = qi.walkers(mol, W, seed=6)
    E, lp, sens = oracle_reference(mol, r)
    sens = _sensitivity(mol, r, sens)
    wf = pkg.Wavefunction(mol, precision="fp32x2")
    e, l = wf.local_energy(torch.tensor(qi.to_soa(r), device="cuda"))
    torch.cuda.synchronize()
    gated_check(e.cpu().numpy(), E, sens)
    wf.close()
