"""Rows of the float64 level-0 product in fixed point (csrc/sym_op.cuh) against
the assembled blocks of agg_dg_mesh_copy in extended precision, each row on its
own: the error of row i relative to (|A| |x|)_i, with conductivity contrasts of
up to 1e8 between neighbours and mass terms large and small, where the diagonal
entries of one element and of its neighbours differ by orders of magnitude.

Tolerance: a float64 sum of T products is off by at most T 2^-53 (|A| |x|)_i;
T = B + 2 d B entries per row at most (T = 448 for Q3 hexahedra). The stored
entries may take 8 2^-53 of a row more (kFxLoss)."""
import numpy as np
import pytest

from paper_2602_16312_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import build
    build.build()


WORKLOADS = {
    "quad_q2": lambda: W.jittered_square_2d(n=9, degree=2, n_levels=2),
    "quad_q3": lambda: W.jittered_square_2d(n=8, degree=3, n_levels=2),
    "hex_q2": lambda: W.jittered_cube_3d(n=4, degree=2, n_levels=2, group=2),
    "hex_q3": lambda: W.cube_3d_adjoint(n=3, degree=3, n_levels=2, n_sensors=1),
    "shell_q2": lambda: W.ventricle_shell(16, 8, 2, degree=2, n_levels=2),
}


def _mesh(wl, contrast):
    from paper_2602_16312_gb300 import aggmg
    D = wl.conductivity.copy()
    D[np.random.default_rng(1).random(len(D)) < 0.3] *= contrast
    return aggmg.Mesh.from_workload(wl, conductivity=D)


class Rows:
    """The rows of c M + A in extended precision: product and (|A| |x|)."""

    def __init__(self, mesh, c):
        rp, cols, vals = mesh.stiffness_bsr()
        me = mesh.element_mass()
        rows = np.repeat(np.arange(mesh.n_elements), np.diff(rp))
        A = vals.copy()
        on = np.nonzero(rows == cols)[0]
        A[on] += c * me[rows[on]]
        self.A, self.rows, self.cols = A.astype(np.longdouble), rows, cols
        self.shape, self.terms = (mesh.n_elements, mesh.B), mesh.B * (1 + 2 * mesh.dim)

    def product(self, x):
        xb = x.reshape(self.shape)[self.cols][:, None, :].astype(np.longdouble)
        y, size = (np.zeros(self.shape, np.longdouble) for _ in range(2))
        np.add.at(y, self.rows, (self.A * xb).sum(2))
        np.add.at(size, self.rows, (np.abs(self.A) * np.abs(xb)).sum(2))
        return y.ravel(), size.ravel()


def _apply(hier, x, level=0):
    y = torch.empty(len(x), dtype=torch.float64, device="cuda")
    hier.operator_apply(level, torch.tensor(x, device="cuda"), y)
    return y.cpu().numpy()


@pytest.mark.parametrize("contrast", [1.0, 1e-2, 1e-4, 1e-8])
@pytest.mark.parametrize("dt", [None, 1000.0])
@pytest.mark.parametrize("kind", sorted(WORKLOADS))
def test_rows_with_contrast(kind, dt, contrast):
    from paper_2602_16312_gb300 import aggmg
    wl = WORKLOADS[kind]()
    mesh = _mesh(wl, contrast)
    c = 1.0 / (wl.dt if dt is None else dt)
    hier = aggmg.Hierarchy(mesh, c, wl.maps, precision="f64")
    ref = Rows(mesh, c)
    for x in (np.random.default_rng(2).standard_normal(wl.n_dofs), np.ones(wl.n_dofs)):
        y, size = ref.product(x)
        for level in (0, -1):
            err = float((np.abs(_apply(hier, x, level) - y) / size).max())
            assert err <= (ref.terms + 8) * 2.0 ** -53, (level, err)
    hier.close()


@pytest.mark.parametrize("contrast,dt", [(1.0, None), (1e-8, 1000.0)])
@pytest.mark.parametrize("kind", sorted(WORKLOADS))
def test_vcycle_with_contrast(kind, contrast, dt):
    """One float64 V-cycle (products with A_0, its block inverses and transfers)
    against the oracle's: 12 products of at most T terms between r and z."""
    from oracle import multigrid as omg
    from oracle import sipg as osipg
    from paper_2602_16312_gb300 import aggmg
    wl = WORKLOADS[kind]()
    D = wl.conductivity.copy()
    D[np.random.default_rng(1).random(len(D)) < 0.3] *= contrast
    c = 1.0 / (wl.dt if dt is None else dt)
    disc = osipg.assemble(wl.mesh.vertices, wl.mesh.elements, D, wl.degree, wl.penalty_mode, wl.penalty_coeff)
    mesh = _mesh(wl, contrast)
    hier = aggmg.Hierarchy(mesh, c, wl.maps, precision="f64")
    r = np.random.default_rng(3).standard_normal(wl.n_dofs)
    z = torch.empty(wl.n_dofs, dtype=torch.float64, device="cuda")
    hier.vcycle_apply(torch.tensor(r, device="cuda"), z)
    ref = omg.vcycle(omg.build_hierarchy(disc, c, wl.maps), r)
    err = float(np.abs(z.cpu().numpy() - ref).max() / np.abs(ref).max())
    assert err <= 12 * mesh.B * (1 + 2 * mesh.dim) * 2.0 ** -53, err
    hier.close()
