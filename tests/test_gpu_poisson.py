"""GPU parity of the Poisson operator, load vector, atom fields and the CEF / CPD / L-CPD
solves against the FP64 CPU oracle, plus closed forms run on the GPU.

Tolerances: operator and fields <= 1e-12 relative (same arithmetic, different order);
solves to relative residual 1e-12 on both sides, compared at 1e-9 relative (the residual
bound times the operator's condition number on these meshes stays below that).
"""
import math

import numpy as np
import pytest
import torch

import workloads as W
from oracle import assembly, poisson, potentials
from oracle.mesh import Mesh as OMesh

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fe():
    import paper_2504_00998_gb300 as fe
    fe.load()
    return fe


def _oracle(slab):
    om = OMesh(slab.L, slab.ncell, slab.p, slab.psi_dirichlet)
    K = assembly.assemble_stiffness(om)
    M = assembly.lumped_mass(om)
    X = om.phi_coords()
    return om, K, M, X


@pytest.mark.parametrize("L,ncell,p", [((4.0, 4.0, 9.0), (2, 2, 4), 3), ((3.0, 5.0, 7.0), (3, 1, 3), 2),
                                       ((6.0, 6.0, 6.0), (2, 2, 2), 6), ((2.0, 2.0, 4.0), (1, 1, 2), 1),
                                       ((12.0, 12.0, 20.0), (6, 6, 10), 4)])
def test_apply_K_matches_oracle(fe, L, ncell, p):
    om = OMesh(L, ncell, p)
    K = assembly.assemble_stiffness(om)
    m = fe.Mesh(L, ncell, p)
    x = np.random.default_rng(0).standard_normal(om.n_phi)
    y = m.poisson_apply_K(torch.tensor(x, device="cuda")).cpu().numpy()
    ref = K @ x
    assert np.linalg.norm(y - ref) / np.linalg.norm(ref) <= 1e-12
    M = assembly.lumped_mass(om)
    np.testing.assert_allclose(m.lumped_mass().cpu().numpy(), M, rtol=1e-14)
    np.testing.assert_allclose(m.node_coords().cpu().numpy(), om.phi_coords(), atol=1e-13)


@pytest.mark.parametrize("L,ncell,p", [((4.0, 4.0, 9.0), (2, 2, 4), 3), ((3.0, 5.0, 7.0), (3, 1, 3), 2),
                                       ((6.0, 6.0, 6.0), (2, 2, 2), 6), ((2.0, 2.0, 4.0), (1, 1, 2), 1),
                                       ((18.0, 4.0, 6.0), (9, 2, 3), 5), ((34.0, 2.0, 4.0), (17, 1, 2), 3),
                                       ((10.0, 6.0, 8.0), (5, 3, 4), 6), ((70.0, 2.0, 4.0), (35, 1, 2), 1),
                                       ((12.0, 12.0, 20.0), (6, 6, 10), 4)])
def test_apply_K_f32_matches_oracle(fe, L, ncell, p):
    """Float K x through the cell-local products (strips of 4 to 32 cells along x, so these
    meshes include partial strips and one-cell periodic directions):
    against the oracle's assembled K on the float-rounded input, 1e-5 relative (float
    accumulation of at most 8 cell contributions of (p+1)-term products); two calls agree
    bit for bit; the float entry rejects aliased arrays."""
    om = OMesh(L, ncell, p)
    K = assembly.assemble_stiffness(om)
    m = fe.Mesh(L, ncell, p)
    x = np.random.default_rng(1).standard_normal(om.n_phi).astype(np.float32)
    xt = torch.tensor(x, device="cuda")
    y1 = m.poisson_apply_K(xt)
    y2 = m.poisson_apply_K(xt)
    assert torch.equal(y1, y2)
    ref = K @ x.astype(np.float64)
    got = y1.double().cpu().numpy()
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-5
    with pytest.raises(fe.FeError):
        fe._lib.call("fe_poisson_apply_K_f32", m.handle, fe._ptr(xt), fe._ptr(xt))


def test_fields_and_load_match_oracle(fe):
    slab = W.small_slab(ncell=(3, 2, 4), p=3, L=(6.0, 4.0, 12.0), natoms=4, seed=11)
    om, K, M, X = _oracle(slab)
    m = fe.Mesh.from_slab(slab)
    f, rho, b = m.poisson_rhs()
    rho_r, b_r = potentials.densities(X, M, slab.R, slab.Z, slab.L)
    np.testing.assert_allclose(rho.cpu().numpy(), rho_r, rtol=1e-12, atol=1e-15)
    np.testing.assert_allclose(b.cpu().numpy(), b_r, rtol=1e-12, atol=1e-15)
    np.testing.assert_allclose(f.cpu().numpy(), 4 * math.pi * M * (rho_r + b_r), rtol=1e-11,
                               atol=1e-14)


@pytest.mark.parametrize("kind", ["cef", "cpd", "lcpd"])
def test_solve_matches_oracle(fe, kind):
    base = W.small_slab(ncell=(3, 3, 6), p=3, L=(6.0, 6.0, 14.0), natoms=3, seed=5)
    bias = {"cef": W.Bias("cef", field=0.02),
            "cpd": W.Bias("cpd", dV=0.03, zA=1.5, zB=12.5),
            "lcpd": W.Bias("cpd", dV=0.03, zA=1.5, zB=12.5, patch=((1.0, 2.0), (4.0, 5.0)))}[kind]
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
    om, K, M, X = _oracle(slab)
    rho, b = potentials.densities(X, M, slab.R, slab.Z, slab.L)
    vl = potentials.vloc_minus_vsm(X, slab.R, slab.Z, slab.L)
    f = 4 * math.pi * M * (rho + b)
    if kind == "cef":
        ref = poisson.solve_cef_direct(K, f, M)
        vapp = potentials.v_app(X[:, 2], bias.field, slab.L[2])
    else:
        mask, vals, om0, om1 = potentials.cpd_constraints(X, vl, bias, slab.L)
        ref = poisson.solve_cpd_direct(K, f, mask, vals)
        vapp = 0.0 * X[:, 2]
    m = fe.Mesh.from_slab(slab)
    phi, vbare, info = m.poisson_solve(bias, rtol=1e-12)
    assert info.status == 0 and info.rel_residual <= 1e-12 and info.iters > 3
    phi = phi.cpu().numpy()
    assert np.max(np.abs(phi - ref)) <= 1e-9 * np.max(np.abs(ref))
    ids = om.psi_to_phi()
    vb_ref = (ref + vl + vapp)[ids]
    assert np.max(np.abs(vbare.cpu().numpy() - vb_ref)) <= 1e-9 * np.max(np.abs(vb_ref))
    if kind == "cef":
        assert abs(M @ phi) <= 1e-10 * np.sum(M) * np.max(np.abs(phi))
    else:
        np.testing.assert_allclose((phi + vl)[om0], 0.0, atol=1e-13)
        np.testing.assert_allclose((phi + vl)[om1], bias.dV, atol=1e-13)


def test_patch_polynomial_and_capacitor_on_gpu(fe):
    """No atoms: rho = -P''/(4 pi) with Dirichlet planes z = 0, Lz reproduces P exactly; with
    rho = 0 the CPD potential is the linear capacitor profile."""
    L, ncell, p = (3.0, 3.0, 8.0), (2, 2, 4), 4
    om = OMesh(L, ncell, p)
    X = om.phi_coords()
    z = X[:, 2]
    m = fe.Mesh(L, ncell, p)
    m.set_atoms(np.zeros((0, 3)), np.zeros(0))
    P = np.polynomial.Polynomial([0.0, 0.4, -0.3, 0.05, 0.01])  # degree p, P(0) = 0
    rho = torch.tensor(-P.deriv(2)(z) / (4 * math.pi), device="cuda")
    bias = W.Bias("cpd", dV=float(P(L[2])), zA=0.0, zB=L[2])
    phi, _, info = m.poisson_solve(bias, rho=rho, rtol=1e-13)
    np.testing.assert_allclose(phi.cpu().numpy(), P(z), atol=1e-10)
    bias = W.Bias("cpd", dV=0.25, zA=2.0, zB=6.0)
    phi, _, info = m.poisson_solve(bias, rho=torch.zeros(om.n_phi, dtype=torch.float64, device="cuda"),
                                   rtol=1e-13)
    np.testing.assert_allclose(phi.cpu().numpy(), np.clip((z - 2.0) / 4.0, 0, 1) * 0.25, atol=1e-11)


def test_iteration_cap_reports_noconv(fe):
    slab = W.small_slab(ncell=(2, 2, 4), p=3, L=(4.0, 4.0, 9.0), natoms=2)
    m = fe.Mesh.from_slab(slab)
    with pytest.raises(fe.FeError) as e:
        m.poisson_solve(slab.bias, rtol=1e-14, max_iter=3)
    assert e.value.status == fe._lib.FE_ENOCONV
    # the mesh stays usable afterwards
    phi, _, info = m.poisson_solve(slab.bias, rtol=1e-10)
    assert info.status == 0


@pytest.mark.parametrize("kind", ["cef", "cpd", "lcpd"])
def test_plane_coarse_space_same_solution_fewer_iterations(fe, kind):
    """The z-plane coarse correction changes only the iteration count: on a long slab
    (4 x 4 x 48 bohr, p = 4) both preconditioners reach the oracle's solution, and the
    two-level one needs clearly fewer iterations."""
    base = W.small_slab(ncell=(2, 2, 24), p=4, L=(4.0, 4.0, 48.0), natoms=4, seed=13)
    bias = {"cef": W.Bias("cef", field=0.01),
            "cpd": W.Bias("cpd", dV=0.05, zA=2.0, zB=46.0),
            "lcpd": W.Bias("cpd", dV=0.05, zA=2.0, zB=46.0, patch=((1.0, 1.0), (3.0, 3.0)))}[kind]
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
    om, K, M, X = _oracle(slab)
    rho, b = potentials.densities(X, M, slab.R, slab.Z, slab.L)
    f = 4 * math.pi * M * (rho + b)
    if kind == "cef":
        ref = poisson.solve_cef_direct(K, f, M)
    else:
        vl = potentials.vloc_minus_vsm(X, slab.R, slab.Z, slab.L)
        mask, vals, _, _ = potentials.cpd_constraints(X, vl, bias, slab.L)
        ref = poisson.solve_cpd_direct(K, f, mask, vals)
    m = fe.Mesh.from_slab(slab)
    iters = {}
    for planes in (False, True):
        m.set_poisson_precond(planes)
        phi, _, info = m.poisson_solve(bias, rtol=1e-12)
        assert info.status == 0 and info.rel_residual <= 1e-12
        assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
        iters[planes] = info.iters
    assert iters[True] < 0.7 * iters[False], iters


@pytest.mark.parametrize("kind", ["cef", "lcpd"])
@pytest.mark.parametrize("layout", ["planes4", "odd_planes", "jacobi_only"])
def test_mixed_refinement_matches_double_cg(fe, kind, layout):
    """Float corrections refined against the double residual reach the double CG's
    solution: same stopping test, solutions within the residual bound times the
    conditioning (1e-9 relative).  Three float iterations are covered: the fused one (planes of
    a multiple of four nodes, plane coarse space), the scalar one (81-node planes) and the
    four-node one without the coarse space (Jacobi only)."""
    p = 3 if layout == "odd_planes" else 4
    base = W.small_slab(ncell=(3, 3, 12), p=p, L=(6.0, 6.0, 24.0), natoms=5, seed=17)
    bias = {"cef": W.Bias("cef", field=0.01),
            "lcpd": W.Bias("cpd", dV=0.05, zA=2.0, zB=22.0, patch=((1.0, 1.0), (4.0, 5.0)))}[kind]
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
    m = fe.Mesh.from_slab(slab)
    if layout == "jacobi_only":
        m.set_poisson_precond(False)
    out = {}
    for mixed in (False, True):
        m.set_poisson_mixed(mixed)
        phi, vb, info = m.poisson_solve(bias, rtol=1e-12)
        assert info.status == 0 and info.rel_residual <= 1e-12
        out[mixed] = phi.cpu().numpy()
    ref = out[False]
    assert np.max(np.abs(out[True] - ref)) <= 1e-9 * np.max(np.abs(ref))


def _bias_for(kind, L):
    Lz = L[2]
    return {"cef": W.Bias("cef", field=0.01),
            "cpd": W.Bias("cpd", dV=0.05, zA=2.0, zB=Lz - 2.0),
            "lcpd": W.Bias("cpd", dV=0.05, zA=2.0, zB=Lz - 2.0,
                           patch=((1.0, 1.0), (0.6 * L[0], 0.7 * L[1])))}[kind]


@pytest.mark.parametrize("kind,p,ncell", [("cef", 4, (3, 3, 12)), ("cpd", 2, (4, 4, 10)),
                                          ("lcpd", 5, (2, 2, 8)), ("cef", 6, (2, 2, 6)),
                                          ("lcpd", 1, (4, 4, 16)), ("cef", 3, (4, 4, 10))])
def test_persistent_cg_matches_launch_per_step(fe, kind, p, ncell):
    """The float CG run as one cooperative kernel per reliable-update interval reaches the
    oracle's solution like the launch-per-step iteration, in about as many iterations
    (the dot products are summed in another order) and with far fewer launches.  p = 1..6,
    the three bias setups, phi planes of 16 to 400 nodes."""
    L = (6.0, 6.0, 24.0)
    base = W.small_slab(ncell=ncell, p=p, L=L, natoms=4, seed=21)
    bias = _bias_for(kind, L)
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
    om, K, M, X = _oracle(slab)
    rho, b = potentials.densities(X, M, slab.R, slab.Z, slab.L)
    f = 4 * math.pi * M * (rho + b)
    if kind == "cef":
        ref = poisson.solve_cef_direct(K, f, M)
    else:
        vl = potentials.vloc_minus_vsm(X, slab.R, slab.Z, slab.L)
        mask, vals, _, _ = potentials.cpd_constraints(X, vl, bias, slab.L)
        ref = poisson.solve_cpd_direct(K, f, mask, vals)
    lib = fe.load()
    m = fe.Mesh.from_slab(slab)
    m.set_poisson_precond(True)   # the plane coarse space on both paths
    out = {}
    for persistent in (False, True):
        m.set_poisson_persistent(persistent)
        n0 = lib.fe_kernel_launches()
        phi, _, info = m.poisson_solve(bias, rtol=1e-12)
        launches = lib.fe_kernel_launches() - n0
        assert info.status == 0 and info.rel_residual <= 1e-12
        phi = phi.cpu().numpy()
        assert np.max(np.abs(phi - ref)) <= 1e-9 * np.max(np.abs(ref))
        out[persistent] = (phi, info.iters, launches)
    it_l, it_p = out[False][1], out[True][1]
    assert abs(it_p - it_l) <= 0.1 * it_l + 3, (it_l, it_p)
    assert out[True][2] < out[False][2] / 3, (out[False][2], out[True][2])


def test_persistent_cg_bounded_wait_reports_timeout(fe):
    """One block of the cooperative CG kernel leaves before its first grid barrier (the test
    aid FE_OPT_TEST_CG_STALL): no barrier can complete, the other blocks' waits run out
    after 2 s, and the solve returns FE_ETIMEOUT instead of hanging; the mesh then solves
    normally."""
    import time
    slab = W.small_slab(ncell=(2, 2, 8), p=4, L=(4.0, 4.0, 16.0), natoms=2, seed=3)
    m = fe.Mesh.from_slab(slab)
    fe.call("fe_set_option", m._h, fe._lib.FE_OPT_TEST_CG_STALL, 1)
    t0 = time.time()
    with pytest.raises(fe.FeError) as e:
        m.poisson_solve(slab.bias, rtol=1e-12)
    assert e.value.status == fe._lib.FE_ETIMEOUT
    assert time.time() - t0 < 60
    fe.call("fe_set_option", m._h, fe._lib.FE_OPT_TEST_CG_STALL, -1)
    phi, _, info = m.poisson_solve(slab.bias, rtol=1e-12)
    assert info.status == 0 and info.rel_residual <= 1e-12
    m.set_poisson_persistent(False)
    phi_l, _, _ = m.poisson_solve(slab.bias, rtol=1e-12)
    ref = phi_l.cpu().numpy()
    assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("p,ncell,L", [(2, (8, 8, 24), (16.0, 16.0, 48.0)),
                                       (3, (8, 12, 12), (16.0, 24.0, 24.0)),
                                       (4, (4, 4, 24), (8.0, 8.0, 48.0))])
def test_mode_coarse_space(fe, p, ncell, L):
    """The plane coarse space enriched with the in-plane modes of wavenumber one: on a CEF
    slab of at least 8 x 8 cells (no constrained phi nodes) the persistent float iteration
    reaches the oracle's solution in clearly fewer iterations than with the plane space
    alone; on a narrower slab, and with constrained nodes (L-CPD), the option acts as the
    plane space (the same iteration count)."""
    base = W.small_slab(ncell=ncell, p=p, L=L, natoms=6, seed=31)
    wide = ncell[0] >= 8 and ncell[1] >= 8
    out = {}
    for kind in ("cef", "lcpd"):
        bias = _bias_for(kind, L)
        slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
        om, K, M, X = _oracle(slab)
        rho, b = potentials.densities(X, M, slab.R, slab.Z, slab.L)
        f = 4 * math.pi * M * (rho + b)
        if kind == "cef":
            ref = poisson.solve_cef_direct(K, f, M)
        else:
            vl = potentials.vloc_minus_vsm(X, slab.R, slab.Z, slab.L)
            mask, vals, _, _ = potentials.cpd_constraints(X, vl, bias, slab.L)
            ref = poisson.solve_cpd_direct(K, f, mask, vals)
        m = fe.Mesh.from_slab(slab)
        for modes in (False, True):
            m.set_poisson_precond(True, modes=modes)
            phi, _, info = m.poisson_solve(bias, rtol=1e-12)
            assert info.status == 0 and info.rel_residual <= 1e-12
            assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
            out[(kind, modes)] = info.iters
    if wide:
        assert out[("cef", True)] < 0.9 * out[("cef", False)], out
    else:
        assert out[("cef", True)] == out[("cef", False)], out
    assert out[("lcpd", True)] == out[("lcpd", False)], out


# n_phi >= 4096 everywhere: chains of 1 to 16 cells, plane sizes off every tile edge, odd planes
@pytest.mark.parametrize("p,ncell", [(1, (16, 16, 16)), (2, (8, 9, 8)), (3, (5, 6, 6)), (4, (1, 8, 8)),
                                     (5, (3, 4, 4)), (6, (3, 3, 3))])
@pytest.mark.parametrize("kind", ["cef", "cpd", "cpd_inside", "lcpd", "lcpd_no_lower_plane"])
def test_separable_preconditioner(fe, kind, p, ncell):
    """The default solve (the separable preconditioner in a double CG) reaches the oracle's
    direct solution, in at most five iterations where whole planes are constrained; a
    constraint set without a separable form (a patch and no constrained plane) still solves,
    and so does a second constraint set on the same mesh.  Bound: the 1e-12 relative residual
    times a condition number below 1e3 relative to the largest value."""
    L = (2.0 * ncell[0] + 1.0, 2.0 * ncell[1] + 1.0, 2.0 * ncell[2] + 6.0)
    Lz = L[2]
    bias = {"cef": W.Bias("cef", field=0.01),
            "cpd": W.Bias("cpd", dV=0.05, zA=0.0, zB=Lz),
            "cpd_inside": W.Bias("cpd", dV=0.05, zA=0.23 * Lz, zB=0.81 * Lz),
            "lcpd": W.Bias("cpd", dV=0.05, zA=0.15 * Lz, zB=0.85 * Lz,
                           patch=((0.1 * L[0], 0.2 * L[1]), (0.6 * L[0], 0.7 * L[1]))),
            "lcpd_no_lower_plane": W.Bias("cpd", dV=0.05, zA=-1.0, zB=0.8 * Lz,
                                          patch=((0.0, 0.2 * L[1]), (0.7 * L[0], 0.9 * L[1])))}[kind]
    base = W.small_slab(ncell=ncell, p=p, L=L, natoms=3, seed=41)
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
    assert slab.n_phi >= 4096
    om, K, M, X = _oracle(slab)
    rho, b = potentials.densities(X, M, slab.R, slab.Z, slab.L)
    vl = potentials.vloc_minus_vsm(X, slab.R, slab.Z, slab.L)
    f = 4 * math.pi * M * (rho + b)
    if kind == "cef":
        ref = poisson.solve_cef_direct(K, f, M)
    else:
        mask, vals, _, _ = potentials.cpd_constraints(X, vl, bias, slab.L)
        ref = poisson.solve_cpd_direct(K, f, mask, vals)
    m = fe.Mesh.from_slab(slab)
    m.poisson_solve(W.Bias("cpd", dV=0.1, zA=0.4 * Lz, zB=0.6 * Lz), rtol=1e-8)
    phi, _, info = m.poisson_solve(bias, rtol=1e-12)
    assert info.status == 0 and info.rel_residual <= 1e-12
    assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))
    if kind in ("cef", "cpd", "cpd_inside"):
        assert info.iters <= 5, info.iters
    elif kind == "lcpd":
        assert info.iters <= 60, info.iters
    with pytest.raises(fe.FeError) as e:
        m.poisson_solve(bias, rtol=1e-12, max_iter=1)
    assert e.value.status == fe._lib.FE_ENOCONV


# z chains of 65 to 129 nodes on planes of 36 to 225 (tiles of 64 and 128 in the z products)
@pytest.mark.parametrize("p,ncell", [(6, (1, 1, 11)), (4, (3, 3, 16)), (1, (11, 12, 64)), (5, (3, 3, 26))])
@pytest.mark.parametrize("kind", ["cef", "cpd"])
def test_separable_long_chains(fe, kind, p, ncell):
    """The default solve on long cells against the oracle's direct one (bounds as above)."""
    L = (2.0 * ncell[0], 2.0 * ncell[1], 1.5 * ncell[2])
    bias = {"cef": W.Bias("cef", field=0.01), "cpd": W.Bias("cpd", dV=0.05, zA=0.0, zB=L[2])}[kind]
    base = W.small_slab(ncell=ncell, p=p, L=L, natoms=3, seed=43)
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, bias)
    om, K, M, X = _oracle(slab)
    rho, b = potentials.densities(X, M, slab.R, slab.Z, slab.L)
    vl = potentials.vloc_minus_vsm(X, slab.R, slab.Z, slab.L)
    f = 4 * math.pi * M * (rho + b)
    if kind == "cef":
        ref = poisson.solve_cef_direct(K, f, M)
    else:
        mask, vals, _, _ = potentials.cpd_constraints(X, vl, bias, slab.L)
        ref = poisson.solve_cpd_direct(K, f, mask, vals)
    phi, _, info = fe.Mesh.from_slab(slab).poisson_solve(bias, rtol=1e-12)
    assert info.status == 0 and info.rel_residual <= 1e-12 and info.iters <= 5
    assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("ncell,p", [((33, 1, 2), 1), ((17, 2, 1), 2), ((16, 3, 2), 3), ((9, 2, 3), 4),
                                     ((8, 1, 2), 5), ((5, 3, 2), 6)])
def test_apply_K_cell_strips(fe, ncell, p):
    """The double stiffness product at full, partial and single strips of cells, with three
    different cell lengths: 1e-12 relative as above, entry by entry 1e-13 of |K| |x|, and two
    calls agree bit for bit."""
    L = (1.3 * ncell[0], 1.9 * ncell[1], 2.6 * ncell[2])
    om = OMesh(L, ncell, p)
    K = assembly.assemble_stiffness(om)
    m = fe.Mesh(L, ncell, p)
    x = np.random.default_rng(p).standard_normal(om.n_phi)
    xt = torch.tensor(x, device="cuda")
    y = m.poisson_apply_K(xt)
    assert torch.equal(y, m.poisson_apply_K(xt))
    y, ref = y.cpu().numpy(), K @ x
    assert np.linalg.norm(y - ref) / np.linalg.norm(ref) <= 1e-12
    assert np.all(np.abs(y - ref) <= 1e-13 * (abs(K) @ np.abs(x)))


def test_captured_product_survives_the_other(fe):
    """A graph around the float product replays correctly after double products and a solve whose
    float iteration refines against them (CEF, Jacobi only: no double product before the
    capture of its iterations)."""
    base = W.small_slab(ncell=(4, 4, 8), p=5, L=(8.0, 8.0, 18.0), natoms=3, seed=7)
    slab = W.Slab(base.name, base.L, base.ncell, base.p, base.R, base.Z, W.Bias("cef", field=0.01))
    om, K, M, X = _oracle(slab)
    s = torch.cuda.Stream()
    m = fe.Mesh(slab.L, slab.ncell, slab.p, stream=s)
    m.set_atoms(slab.R, slab.Z)
    m.set_poisson_precond(False)
    x = torch.tensor(np.random.default_rng(2).standard_normal(om.n_phi).astype(np.float32), device="cuda")
    ref = K @ x.double().cpu().numpy()
    y = torch.zeros_like(x)
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        m.poisson_apply_K(x, y)
        g = torch.cuda.CUDAGraph()
        s.synchronize()
        with torch.cuda.graph(g, stream=s):
            m.poisson_apply_K(x, y)
        phi, _, info = m.poisson_solve(slab.bias, rtol=1e-12)
        m.poisson_apply_K(x.double())
        y.zero_()
        g.replay()
    s.synchronize()
    assert info.status == 0
    assert np.linalg.norm(y.double().cpu().numpy() - ref) / np.linalg.norm(ref) <= 1e-5
    f = 4 * math.pi * M * sum(potentials.densities(X, M, slab.R, slab.Z, slab.L))
    phi_ref = poisson.solve_cef_direct(K, f, M)
    assert np.max(np.abs(phi.cpu().numpy() - phi_ref)) <= 1e-9 * np.max(np.abs(phi_ref))


def test_double_cg_captures_the_cell_product(fe):
    """FE_POISSON_F64 runs the same products in its captured iterations whether or not one was
    made before (its scratch is taken before the capture): bitwise equal potentials."""
    base = W.small_slab(ncell=(3, 3, 8), p=4, L=(6.0, 6.0, 18.0), natoms=3, seed=7)
    bias = W.Bias("cef", field=0.01)
    out = []
    for warm in (False, True):
        m = fe.Mesh.from_slab(base)
        m.set_poisson_precond(False)
        m.set_poisson_mixed(False)
        if warm:
            m.poisson_apply_K(torch.ones(m.n_phi, dtype=torch.float64, device="cuda"))
        phi, _, info = m.poisson_solve(bias, rtol=1e-12)
        assert info.status == 0
        out.append(phi)
    assert torch.equal(out[0], out[1])


# loads inside the floats' range, above it, and below it
@pytest.mark.parametrize("scale", [1e25, 1e42, 1e-30, 1e-46])
@pytest.mark.parametrize("kind", ["cef", "cpd"])
def test_default_solve_of_scaled_loads(fe, kind, scale):
    """The problem is linear: a load outside the range of the float preconditioner is handed to
    the other iterations and solved, with the bound of test_separable_preconditioner."""
    L = (9.0, 9.0, 14.0)
    om = OMesh(L, (4, 4, 4), 4)
    K, M = assembly.assemble_stiffness(om), assembly.lumped_mass(om)
    f = np.random.default_rng(3).standard_normal(om.n_phi) * M
    assert om.n_phi >= 4096
    m = fe.Mesh(L, (4, 4, 4), 4)
    m.set_atoms(np.zeros((0, 3)), np.zeros(0))
    if kind == "cef":
        bias = W.Bias("cef", field=0.01)
        ref = poisson.solve_cef_direct(K, f, M)
    else:
        bias = W.Bias("cpd", dV=0.0, zA=0.0, zB=L[2])
        mask = m.poisson_constraints(bias)[0].cpu().numpy()
        ref = poisson.solve_cpd_direct(K, f, mask, np.zeros(om.n_phi))
    phic = None if kind == "cef" else torch.zeros(om.n_phi, dtype=torch.float64, device="cuda")
    phi, info = m.poisson_solve_load(torch.tensor(scale * f, device="cuda"), bias, phic=phic, rtol=1e-12)
    assert info.status == 0 and info.rel_residual <= 1e-12
    assert np.max(np.abs(phi.cpu().numpy() / scale - ref)) <= 1e-9 * np.max(np.abs(ref))


# smooth load on a long chain: rounding of K phi stays far above the recurrence's last residual
@pytest.mark.parametrize("p,ncell,rtol", [(4, (4, 4, 40), 1e-10), (5, (3, 3, 30), 1e-11), (6, (3, 3, 24), 1e-10)])
def test_default_solve_reports_the_residual_of_phi(fe, p, ncell, rtol):
    """rel_residual of the default solve is that of the returned potential, |f - K phi| over the
    free nodes relative to its value at the start, to a tenth."""
    L = (2.0 * ncell[0], 2.0 * ncell[1], 2.0 * ncell[2])
    m = fe.Mesh(L, ncell, p)
    m.set_atoms(np.zeros((0, 3)), np.zeros(0))
    X = m.node_coords()
    f = m.lumped_mass() * torch.sin(math.pi * X[:, 2] / L[2])
    bias = W.Bias("cpd", dV=0.5, zA=0.0, zB=L[2])
    mask, vals = m.poisson_constraints(bias)
    phi, info = m.poisson_solve_load(f, bias, phic=vals, rtol=rtol)
    assert info.status == 0 and info.rel_residual <= rtol

    def residual(x):
        return torch.linalg.vector_norm((f - m.poisson_apply_K(x))[~mask]).item()

    true = residual(phi) / residual(torch.where(mask, vals, torch.zeros_like(vals)))
    assert abs(info.rel_residual - true) <= 0.1 * true, (info.rel_residual, true)


# cells far longer in one direction than in the others: the slowest mode along it is 2e-11 to 3e-11
# of the largest eigenvalue
@pytest.mark.parametrize("p,ncell,h", [(4, (2, 2, 127), (0.01, 0.01, 2.0)), (2, (3, 3, 250), (1.0, 0.005, 2.0)),
                                       (3, (170, 2, 2), (2.0, 0.005, 0.005))])
def test_separable_unequal_cells(fe, p, ncell, h):
    """The default solve keeps its few iterations on very unequal cell lengths: no mode but the
    constant is dropped.  Two modes of 18,000 to 33,000 hold 1e-2 of a random load, eps / 2e-11
    times that is the rounding of K phi; rtol lies between."""
    L = tuple(n * d for n, d in zip(ncell, h))
    m = fe.Mesh(L, ncell, p)
    m.set_atoms(np.zeros((0, 3)), np.zeros(0))
    f = m.lumped_mass() * torch.tensor(np.random.default_rng(9).standard_normal(m.n_phi), device="cuda")
    phi, info = m.poisson_solve_load(f, W.Bias("cef", field=0.0), rtol=1e-4)
    assert info.status == 0 and info.iters <= 6, info.iters


def test_default_preconditioner_can_be_set_again(fe):
    """After another preconditioner the default one comes back: the same iterations and bits as
    on a fresh mesh; values without a meaning stay refused."""
    base = W.small_slab(ncell=(4, 4, 8), p=3, L=(8.0, 8.0, 18.0), natoms=3, seed=7)
    bias = W.Bias("cef", field=0.01)
    m = fe.Mesh.from_slab(base)
    phi, _, info = m.poisson_solve(bias, rtol=1e-12)
    m.set_poisson_precond(True, modes=True)
    other = m.poisson_solve(bias, rtol=1e-12)[2].iters
    m.reset_poisson_precond()
    again, _, info2 = m.poisson_solve(bias, rtol=1e-12)
    assert info2.iters == info.iters < other and torch.equal(phi, again)
    for value in (-1, 4):
        with pytest.raises(fe.FeError):
            fe.call("fe_set_option", m.handle, fe._lib.FE_OPT_POISSON_PRECOND, value)
