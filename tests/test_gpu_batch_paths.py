"""Batched mixed-precision calls on the paths chosen by size: the assembled FP32 operator's
splits of a row (by the number of columns) and the starts from a basis of the call's own
solutions.  The reference is the FP64 solve; mixed results differ from it by the rounding of
the element data, about 1e-7 relative, and 1e-6 bounds that."""
import numpy as np
import pytest

import rve_inputs as ri

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rve():
    import paper_1610_03484_gb300 as pkg
    from paper_1610_03484_gb300 import _build
    _build.build()
    pkg.load_library()
    return pkg


def tensors(rve, grid, p, T, c, t, bc, **opts):
    xyz, tets, phase, tangent = ri.weave_rve(*grid)
    with rve.Context(**opts) as ctx:
        m = ctx.mesh_load(xyz, tets, p, phase, tangent)
        m.set_materials(ri.NOMINAL_MATRIX, ri.NOMINAL_YARN)
        m.set_bc(bc)
        C, K, D, status, stats, rc = ctx.macro_update([m], T, c, t, np.zeros(len(T), np.int32))
        m.free()
    assert rc == 0 and (status == 0).all()
    return (C, K, D), stats


def close(got, want, tol=1e-6):
    for a, b in zip(got, want):
        n = len(a)
        err = np.linalg.norm((a - b).reshape(n, -1), axis=1) / np.linalg.norm(b.reshape(n, -1), axis=1)
        assert err.max() < tol, err.max()


@pytest.mark.parametrize("batch", [1, 2, 3, 4, 9, 40])
def test_assembled_row_splits(rve, batch):
    """6, 12, 18, 24, 54 and 240 columns; a last batch of another size."""
    T, c, t, _, _ = ri.gauss_point_states(batch + 1, 3)
    args = ((7, 6, 5), 1, T, c, t, rve.BC_PERIODIC)
    got, _ = tensors(rve, *args, precision=rve.PREC_MIXED, rtol=1e-8, batch=batch)
    want, _ = tensors(rve, *args, precision=rve.PREC_FP64, rtol=1e-10, batch=batch)
    close(got, want)


@pytest.mark.parametrize("grid,p,points,batch,spread", [
    ((9, 9, 5), 2, 60, 7, "wide"),       # ragged last batch
    ((9, 9, 5), 2, 60, 7, "equal"),      # one factor: parallel sources
    ((9, 9, 5), 2, 53, 6, "two"),        # two factors; the fewest points of the rule, whole batches
    ((16, 15, 6), 1, 121, 64, "wide"),
    ((5, 5, 4), 3, 66, 16, "wide"),      # element operators
])
def test_starts_from_a_basis(rve, grid, p, points, batch, spread):
    rng = np.random.default_rng(points)
    T, c = np.full(points, 60.0), np.full(points, 1.5)
    t = {"wide": 10.0 ** rng.uniform(0, 4.3, points), "equal": np.full(points, 3000.0),
         "two": np.where(np.arange(points) % 2, 10.0, 9000.0)}[spread]
    for bc in (rve.BC_PERIODIC, rve.BC_DIRICHLET):
        got, stats = tensors(rve, grid, p, T, c, t, bc, precision=rve.PREC_MIXED, rtol=1e-5, batch=batch)
        assert stats["rel_residual_mech"] <= 1e-5
        want, _ = tensors(rve, grid, p, T, c, t, bc, precision=rve.PREC_FP64, rtol=1e-9, batch=batch)
        close(got, want)
