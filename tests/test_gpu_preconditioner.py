"""The polynomial preconditioner of the FP64 solves away from regular meshes and data."""
import numpy as np
import pytest

import rve_inputs as ri
from oracle import fem
from oracle import macro as mo
from oracle import materials as mt

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rve():
    import paper_1610_03484_gb300 as pkg
    from paper_1610_03484_gb300 import _build
    _build.build()
    pkg.load_library()
    return pkg


def isotropic(E=1.0, nu=0.3):
    la, mu = E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))
    C = np.zeros((6, 6))
    C[:3, :3] = la
    C[range(3), range(3)] += 2 * mu
    C[range(3, 6), range(3, 6)] = mu
    return C


def plate_solve(rve, xyz, tets, C, rtol, max_iter, traction=(1e-3, 0.0, 0.0)):
    """(stats, u, load) of a plate on rollers under a traction on its far end"""
    with rve.Context() as ctx:
        m = ctx.macro_load(xyz, tets)
        m.mech_set_bc(xyz <= 1e-12)
        m.mech_set_traction(xyz[:, 0] >= xyz[:, 0].max() * (1 - 1e-12), list(traction))
        st = m.mech_solve(C, rtol=rtol, max_iter=max_iter)
        r = m.mech_get()
        m.free()
    return st, r["u"], r["load"]


def residual(xyz, tets, C, u, load):
    """sqrt((r, D^-1 r) / (f, D^-1 f)) over the free DOFs"""
    K = mo.elastic_assemble(xyz, tets, C)
    free = ~(xyz <= 1e-12).reshape(-1)
    f, d = load.reshape(-1)[free], K.diagonal()[free]
    r = f - (K @ u.reshape(-1))[free]
    return np.sqrt((r @ (r / d)) / (f @ (f / d)))


def test_eigenvalue_above_the_estimate(rve):
    """One tetrahedron 16 times as stiff, placed where the power iteration's start hardly
    sees it: the largest eigenvalue of D^-1 K is 2.80, the estimate 2.75 (both by
    arithmetic on the host).  49 665 nodes, for which sqrt(ratio) rounds to 32: a polynomial
    of that degree is indefinite and takes 1364 iterations, where the uniform plate takes
    36 and Jacobi preconditioning 904."""
    grid = (104, 42, 10)
    xyz, tets = ri.kuhn_grid(*grid, tuple(float(g) for g in grid))
    C = np.broadcast_to(isotropic(), (len(tets), 4, 6, 6)).copy()
    C[247260] *= 16.0
    st, u, load = plate_solve(rve, xyz, tets, C, 1e-10, 250)
    assert st["converged"] == 1
    # (the recurrence's residual and the true one part at rounding level)
    assert residual(xyz, tets, C, u, load) < 2e-10


def distorted(grid, seed, amp=0.25):
    """the box with its interior nodes displaced by up to amp cells"""
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    rng = np.random.default_rng(seed)
    inner = ((xyz > 1e-9) & (xyz < xyz.max(0) - 1e-9)).all(1)
    xyz = xyz.copy()
    xyz[inner] += amp * rng.uniform(-1, 1, (inner.sum(), 3)) * (xyz.max(0) / np.array(grid)) / 2
    return xyz, tets, phase, tangent


@pytest.mark.parametrize("grid,p", [((3, 3, 2), 1), ((3, 3, 3), 1), ((3, 3, 4), 1), ((6, 6, 4), 1), ((9, 8, 6), 1),
                                    ((5, 4, 3), 2), ((3, 3, 2), 3)])
def test_distorted_cells_match_oracle(rve, grid, p):
    xyz, tets, phase, tangent = distorted(grid, 3)
    mat, yarn = ri.NOMINAL_MATRIX, ri.NOMINAL_YARN
    D, K, Dd = mt.element_tensors(phase, tangent, mat, yarn, w_matrix=float(mt.one_minus_omega(45.0, 1.0, 800.0)))
    want = fem.homogenise(xyz, tets, grid, p, rve.BC_DIRICHLET, D, K, Dd)
    with rve.Context(precision=rve.PREC_FP64, rtol=1e-11) as ctx:
        m = ctx.mesh_load(xyz, tets, p, phase, tangent)
        m.set_materials(mat, yarn, T_C=45.0, c_wt=1.0, t_h=800.0)
        m.set_bc(rve.BC_DIRICHLET)
        r = m.homogenise()
        m.free()
    for got, ref in zip((r.C, r.K, r.D), want):
        assert np.linalg.norm(got - ref) < 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("grid,p,bc", [((5, 4, 3), 1, 1), ((4, 3, 2), 2, 1), ((4, 3, 2), 2, 0), ((3, 3, 2), 3, 0)])
def test_degradation_factor_below_fp32(rve, grid, p, bc):
    """Factors whose FP32 value is subnormal or zero, alone and among others in one batch:
    the tensors approach those of a vanishing matrix (1e-20 already agrees to 1e-12)."""
    W = np.array([0.7, 1e-20, 1e-37, 1e-39, 1e-42, 1e-60])
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    with rve.Context(precision=rve.PREC_FP64, rtol=1e-9) as ctx:
        m = ctx.mesh_load(xyz, tets, p, phase, tangent)
        m.set_materials(ri.NOMINAL_MATRIX, ri.NOMINAL_YARN)
        m.set_bc(bc)
        batch = ctx.macro_update_w([m], W, np.zeros(len(W), np.int32))
        single = [ctx.macro_update_w([m], W[i:i + 1], np.zeros(1, np.int32)) for i in range(len(W))]
        m.free()
    assert (batch[3] == 0).all()
    for i in range(len(W)):
        C = single[i][0][0]
        assert np.linalg.norm(batch[0][i] - C) < 1e-10 * np.linalg.norm(C)
        if i > 0:
            ref = single[1][0][0]
            assert np.linalg.norm(C - ref) < 1e-10 * np.linalg.norm(ref)


@pytest.mark.parametrize("grid,p", [((4, 4, 2), 1), ((5, 4, 3), 2)])
def test_uniform_traction_at_rounding_level(rve, grid, p):
    """A tolerance at rounding level, which the unconstrained (singular) start of the uniform
    traction cannot reach: the constrained solve decides, and answers as at 1e-13."""
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    out = []
    for rtol in (1e-13, 3e-16):
        with rve.Context(precision=rve.PREC_FP64, rtol=rtol) as ctx:
            m = ctx.mesh_load(xyz, tets, p, phase, tangent)
            m.set_materials(ri.NOMINAL_MATRIX, ri.NOMINAL_YARN, T_C=40.0, c_wt=1.0, t_h=2000.0)
            m.set_bc(rve.BC_NEUMANN)
            out.append(m.homogenise())
            m.free()
    for a, b in ((out[0].C, out[1].C), (out[0].K, out[1].K), (out[0].D, out[1].D)):
        assert np.linalg.norm(a - b) < 1e-11 * np.linalg.norm(a)


@pytest.mark.parametrize("grid,p,batch", [((4, 4, 3), 1, 3), ((4, 3, 2), 2, 2), ((3, 2, 2), 3, 4)])
def test_uniform_traction_batches(rve, grid, p, batch):
    """Several factors a batch: each RVE's own multipliers; against one call per factor in
    the mixed precision of the same context, whose solves take no such start (1e-6: the
    rounding of its element data)."""
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    W = np.linspace(1.0, 0.2, 2 * batch + 1)
    res = []
    for prec, b, rtol in ((rve.PREC_FP64, batch, 1e-11), (rve.PREC_MIXED, 1, 1e-9)):
        with rve.Context(precision=prec, rtol=rtol, batch=b, warm_start=0) as ctx:
            m = ctx.mesh_load(xyz, tets, p, phase, tangent)
            m.set_materials(ri.NOMINAL_MATRIX, ri.NOMINAL_YARN)
            m.set_bc(rve.BC_NEUMANN)
            res.append(ctx.macro_update_w([m], W, np.zeros(len(W), np.int32)))
            m.free()
    assert (res[0][3] == 0).all()
    for a, b in zip(res[0][:3], res[1][:3]):
        for i in range(len(W)):
            assert np.linalg.norm(a[i] - b[i]) < 1e-6 * np.linalg.norm(b[i]), i


@pytest.mark.parametrize("grid,p", [((6, 6, 4), 1), ((4, 4, 3), 2)])
def test_one_mesh_through_many_materials(rve, grid, p):
    """What a mesh keeps from solve to solve (matrix entries, the spectrum's estimate, the
    captured loop) against a fresh mesh for every call: new constituents, the same ones in
    another state, boundary conditions with and without a change of the DOF map."""
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    a = (ri.NOMINAL_MATRIX, ri.NOMINAL_YARN)
    b = ri.jitter_props(5)
    c = ri.jitter_props(6, frac=0.4)
    calls = [(a, 40.0, 500.0, 1), (b, 40.0, 500.0, 1), (b, 60.0, 9000.0, 1), (b, 60.0, 9000.0, 0), (b, 60.0, 9000.0, 2),
             (c, 60.0, 9000.0, 2), (c, 60.0, 100.0, 0), (a, 40.0, 500.0, 1), (a, 40.0, 500.0, 1)]
    with rve.Context(precision=rve.PREC_FP64, rtol=1e-11) as ctx:
        kept = ctx.mesh_load(xyz, tets, p, phase, tangent)
        for props, T, t, bc in calls:
            got = []
            for m in (kept, ctx.mesh_load(xyz, tets, p, phase, tangent)):
                m.set_materials(*props, T_C=T, c_wt=1.0, t_h=t)
                m.set_bc(bc)
                got.append(m.homogenise())
            m.free()
            for x, y in ((got[0].C, got[1].C), (got[0].K, got[1].K), (got[0].D, got[1].D)):
                assert np.linalg.norm(x - y) < 1e-11 * np.linalg.norm(y)
            assert abs(got[0].stats["iterations_mech"] - got[1].stats["iterations_mech"]) <= 1
        kept.free()


@pytest.mark.parametrize("grid,p,bc", [((6, 6, 4), 1, 1), ((5, 5, 4), 2, 0), ((3, 3, 2), 3, 1)])
def test_profile_counts_the_preconditioners_products(rve, grid, p, bc):
    """FP64 in profile mode: an iteration is one FP64 product and the polynomial's FP32
    products (degree 5 at these sizes: four), all operator launches; their time is the
    operator's, not the update pass's."""
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    with rve.Context(precision=rve.PREC_FP64, rtol=1e-10, profile=1) as ctx:
        m = ctx.mesh_load(xyz, tets, p, phase, tangent)
        m.set_materials(ri.NOMINAL_MATRIX, ri.NOMINAL_YARN, T_C=40.0, c_wt=1.0, t_h=500.0)
        m.set_bc(bc)
        m.homogenise()
        st = m.homogenise().stats
        m.free()
    n = st["iterations_mech"] + st["iterations_scalar"]
    assert st["op_launches"] == 5 * n
    # one pass over at most 9 vectors, against five products: some slack for launch gaps
    assert st["update_ms"] < 0.7 * st["op_ms"]


@pytest.mark.parametrize("grid,p,bc,prec", [((6, 6, 4), 1, 1, 0), ((5, 4, 3), 2, 0, 0), ((5, 4, 3), 2, 2, 0),
                                            ((16, 15, 6), 1, 1, 1), ((24, 20, 10), 1, 1, 0),
                                            ((12, 11, 8), 2, 0, 0)])
def test_matrix_without_room(rve, grid, p, bc, prec):
    """No room for the matrix' entries: the element operators answer, as before there was a
    matrix; and with room again the matrix does."""
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    W = np.linspace(1.0, 0.3, 18 if prec else 2)
    res = []
    with rve.Context(precision=prec, rtol=1e-9, batch=18 if prec else 2) as ctx:
        m = ctx.mesh_load(xyz, tets, p, phase, tangent)
        m.set_materials(ri.NOMINAL_MATRIX, ri.NOMINAL_YARN)
        m.set_bc(bc)
        for limit in (0, 1000, 0):
            m.debug_set_matrix_limit(limit)
            res.append(ctx.macro_update_w([m], W, np.zeros(len(W), np.int32)))
        m.free()
    tol = 1e-6 if prec else 1e-12   # (mixed: FP32 element data against an FP32 matrix)
    for other in res[1:]:
        assert (other[3] == 0).all()
        for a, b in zip(res[0][:3], other[:3]):
            assert np.linalg.norm(a - b) < tol * np.linalg.norm(b)
    assert res[1][4]["kernel_launches"] != res[0][4]["kernel_launches"]


@pytest.mark.parametrize("stiffness,force", [(1.0, 1e-60), (1.0, 1e60), (1e11, 1e-40), (1e45, 1e45), (1e-45, 1e-45)])
def test_plate_in_any_units(rve, stiffness, force):
    """The same plate with the stiffness and the traction in other units: the displacement
    scales with force / stiffness.  Residuals far outside FP32's range, and (last two) a
    matrix outside it, where the Jacobi iteration has to take over."""
    xyz, tets = ri.kuhn_grid(9, 4, 3, (9.0, 4.0, 3.0))
    C = np.broadcast_to(isotropic(), (len(tets), 4, 6, 6))
    st0, u0, _ = plate_solve(rve, xyz, tets, C, 1e-11, 2000)
    st, u, load = plate_solve(rve, xyz, tets, C * stiffness, 1e-11, 2000, (1e-3 * force, 0.0, 0.0))
    assert st["converged"] == 1 and st["rel_residual"] <= 1e-11
    if abs(np.log10(stiffness)) < 38:
        assert st["iterations"] <= st0["iterations"] + 1
    want = u0 * (force / stiffness)
    assert np.linalg.norm(u - want) < 1e-9 * np.linalg.norm(want)


def test_not_a_number_does_not_read_as_converged(rve):
    xyz, tets = ri.kuhn_grid(5, 3, 2, (5.0, 3.0, 2.0))
    C = np.broadcast_to(isotropic(), (len(tets), 4, 6, 6)).copy()
    C[len(tets) // 2, 0, 0, 0] = np.nan
    with pytest.raises(rve.RveError) as e:
        plate_solve(rve, xyz, tets, C, 1e-11, 500)
    assert e.value.code == -4


def limit_matrices(ctx, m, n_bytes):
    assert ctx.lib.rve_debug_macro_matrix_limit(ctx.h, m.h, n_bytes) == 0


def test_macro_mesh_without_room_for_matrices(rve):
    """No room for the graph and the matrices: transport steps and the elastic solve element by
    element, against the matrices and, for the displacements, the oracle."""
    rng = np.random.default_rng(4)
    xyz, tets, _ = ri.plate(9, 4, 3)
    A = rng.standard_normal((len(tets), 4, 6, 6))
    C = 1e9 * (np.einsum("tgij,tgkj->tgik", A, A) + 6 * np.eye(6))
    KT = np.array([[0.40, 0.01, 0.0], [0.01, 0.35, 0.0], [0.0, 0.0, 0.30]])
    out = []
    with rve.Context() as ctx:
        m = ctx.macro_load(xyz, tets)
        m.set_face(xyz[:, 2] <= 1e-12, 60.0, 1.5)
        m.mech_set_bc(xyz <= 1e-12)
        m.mech_set_traction(xyz[:, 0] >= xyz[:, 0].max() * (1 - 1e-12), [1e6, 0.0, 2e5])
        for limit in (0, 100, 0):   # one mesh, back and forth
            limit_matrices(ctx, m, limit)
            m.set_transport(KT, 1.6e6, np.diag([1.2e-12, 1.0e-12, 8.0e-13]))
            m.reset(20.0, 0.1)
            for dt in (50.0, 50.0, 20.0):
                m.step(dt)
            m.mech_set_u(None)
            m.mech_solve(C, rtol=1e-12)
            g, r = m.get(), m.mech_get()
            out.append([np.asarray(v) for v in (g["T"], g["c"], g["W"], r["u"], r["stress"])])
        m.free()
    for other in out[1:]:
        for a, b in zip(out[0], other):
            assert np.linalg.norm(a - b) < 1e-9 * np.linalg.norm(a)
    K = mo.elastic_assemble(xyz, tets, C)
    u = mo.elastic_solve(K, r["load"].reshape(-1), (xyz <= 1e-12).reshape(-1))
    for o in out:
        assert np.linalg.norm(o[3].reshape(-1) - u) < 1e-9 * np.linalg.norm(u)


def test_macro_mesh_with_a_hub(rve):
    """A fan of tetrahedra around one edge: its two nodes couple to all others, and slices of
    equal row length would be mostly padding.  Answered element by element."""
    n = 2400
    phi = 2 * np.pi * np.arange(n) / n
    xyz = np.concatenate([[[0, 0, -0.5], [0, 0, 0.5]], np.stack([np.cos(phi), np.sin(phi), 0 * phi], 1)])
    i = np.arange(n)
    tets = np.stack([0 * i, 0 * i + 1, 2 + i, 2 + (i + 1) % n], 1).astype(np.int32)
    X = xyz[tets]
    if np.linalg.det(X[0, 1:] - X[0, 0]) < 0:
        tets = tets[:, [1, 0, 2, 3]]
    C = np.broadcast_to(isotropic(1e3), (len(tets), 4, 6, 6)).copy()
    fixed = np.zeros((len(xyz), 3), bool)
    fixed[2::3] = True
    with rve.Context() as ctx:
        m = ctx.macro_load(xyz, tets)
        m.mech_set_bc(fixed)
        m.mech_set_traction(np.arange(len(xyz)) != 0, [0.0, 1.0, 3.0])
        m.mech_solve(C, rtol=1e-12)
        r = m.mech_get()
        m.free()
    u = mo.elastic_solve(mo.elastic_assemble(xyz, tets, C), r["load"].reshape(-1), fixed.reshape(-1))
    assert np.linalg.norm(u) > 0
    assert np.linalg.norm(r["u"].reshape(-1) - u) < 1e-9 * np.linalg.norm(u)
