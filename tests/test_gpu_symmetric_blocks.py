"""The symmetric level-0 blocks (csrc/sym_op.cuh): the fixed-point float64
product and the V-cycle on them, at element counts around the tiles of the
kernels, over the range of magnitudes, with NaN and infinities, and the
face-structured form that an unsymmetric conductivity keeps. Reference: the
product with the assembled blocks of agg_dg_mesh_copy in numpy float64.

Tolerance of the products: both sides round a sum of at most 304 products, in
units of the row's largest neighbour value (elements of one mesh size), so
304 * 2^-53 = 3.4e-14 of max |y|; 1e-13 is used."""
import numpy as np
import pytest

from paper_2602_16312_gb300 import workloads as W

from gpu_util import rel

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import build
    build.build()


def _product(mesh, c):
    """x -> (c M + A) x and the dense coupling test (rows coupled to a DoF)."""
    rp, cols, vals = mesh.stiffness_bsr()
    me = mesh.element_mass()
    B = mesh.B
    rows = np.repeat(np.arange(mesh.n_elements), np.diff(rp))

    def apply(x):
        xb = x.reshape(-1, B)
        y = c * np.einsum("eij,ej->ei", me, xb)
        np.add.at(y, rows, np.einsum("kij,kj->ki", vals, xb[cols]))
        return y.ravel()

    def coupled(dof):
        e, j = divmod(dof, B)
        out = np.zeros((mesh.n_elements, B), bool)
        for k in np.nonzero(cols == e)[0]:
            out[rows[k]] |= vals[k][:, j] != 0.0
        out[e] = True
        return out.ravel()
    return apply, coupled


CASES = [("jsquare", 5, 3), ("jsquare", 7, 3), ("jsquare", 4, 2), ("jsquare", 7, 2), ("jsquare", 5, 1),
         ("jcube", 2, 2), ("jcube", 4, 2), ("jcube", 5, 2), ("jcube", 3, 1), ("jcube", 2, 3), ("jcube", 3, 3),
         ("shell", 16, 2)]


def _workload(kind, n, p):
    if kind == "jsquare":
        return W.jittered_square_2d(n=n, degree=p, n_levels=2)
    if kind == "jcube":
        return W.jittered_cube_3d(n=n, degree=p, n_levels=2, group=2)
    return W.ventricle_shell(n, 8, 2, degree=p, n_levels=2)


@pytest.mark.parametrize("scale", [1.0, 1e-250, 1e250])
@pytest.mark.parametrize("kind,n,p", CASES)
def test_float64_product(kind, n, p, scale):
    from paper_2602_16312_gb300 import aggmg
    wl = _workload(kind, n, p)
    mesh = aggmg.Mesh.from_workload(wl)
    hier = aggmg.Hierarchy(mesh, 1.0 / wl.dt, wl.maps, precision="f64")
    apply, _ = _product(mesh, 1.0 / wl.dt)
    x = np.random.default_rng(4).standard_normal(wl.n_dofs) * scale
    y = torch.empty(wl.n_dofs, dtype=torch.float64, device="cuda")
    for level in (0, -1):
        hier.operator_apply(level, torch.tensor(x, device="cuda"), y)
        assert rel(y.cpu().numpy() / scale, apply(x / scale)) <= 1e-13
    hier.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("kind,n,p", [("jsquare", 5, 3), ("jcube", 3, 2), ("jcube", 2, 3)])
def test_nan_and_infinity_reach_the_coupled_rows_only(kind, n, p, bad):
    from paper_2602_16312_gb300 import aggmg
    wl = _workload(kind, n, p)
    mesh = aggmg.Mesh.from_workload(wl)
    hier = aggmg.Hierarchy(mesh, 1.0 / wl.dt, wl.maps, precision="f64")
    apply, coupled = _product(mesh, 1.0 / wl.dt)
    x = np.random.default_rng(5).standard_normal(wl.n_dofs)
    ref = apply(x)
    dof = wl.n_dofs // 2 + 1
    x[dof] = bad
    y = torch.empty(wl.n_dofs, dtype=torch.float64, device="cuda")
    hier.operator_apply(0, torch.tensor(x, device="cuda"), y)
    y = y.cpu().numpy()
    hit = coupled(dof)
    assert not np.isfinite(y[hit]).any()
    assert np.abs(y[~hit] - ref[~hit]).max() <= 1e-13 * np.abs(ref).max()
    r = torch.tensor(x, device="cuda")
    res = hier.pcg_solve(r, torch.zeros_like(r), check=False)
    assert res["status"] == aggmg.AGG_ENAN
    hier.close()


@pytest.mark.parametrize("kind,n,p", [("jsquare", 5, 2), ("jsquare", 4, 3), ("jcube", 3, 2)])
def test_unsymmetric_conductivity_keeps_its_product(kind, n, p):
    from paper_2602_16312_gb300 import aggmg
    wl = _workload(kind, n, p)
    D = wl.conductivity.copy()
    D[:, 0, 1] *= 1.05
    mesh = aggmg.Mesh.from_workload(wl, conductivity=D)
    hier = aggmg.Hierarchy(mesh, 1.0 / wl.dt, wl.maps, precision="f64")
    apply, _ = _product(mesh, 1.0 / wl.dt)
    x = np.random.default_rng(6).standard_normal(wl.n_dofs)
    y = torch.empty(wl.n_dofs, dtype=torch.float64, device="cuda")
    hier.operator_apply(0, torch.tensor(x, device="cuda"), y)
    assert rel(y.cpu().numpy(), apply(x)) <= 1e-13
    hier.close()
