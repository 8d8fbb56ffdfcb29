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


def _vectors(wl, rng):
    """Vectors whose values differ by many orders of magnitude, within elements
    and from element to element."""
    n, B = wl.n_dofs, (wl.degree + 1) ** wl.mesh.dim
    N = wl.degree + 1
    index = np.arange(B)
    inner = np.ones(B, bool)
    for k in range(wl.mesh.dim):
        i = index // N ** k % N
        inner &= (i > 0) & (i < N - 1)
    noise = rng.standard_normal(n)
    centre = wl.mesh.vertices[wl.mesh.elements].mean(1)
    dist = np.linalg.norm(centre - centre[0], axis=1)
    steps = dist / np.sort(dist)[1]
    out = {}
    mid = n // B // 2 * B
    for name, dof in (("corner", 0), ("inner", int(index[inner][0]))):
        out["unit_" + name] = np.eye(1, n, mid + dof)[0]
        for tiny in (1e-2, 1e-4, 1e-12, 1e-30):
            out[f"unit_{name}_over_{tiny}"] = np.eye(1, n, mid + dof)[0] + tiny * noise
    out["decay"] = noise * 10.0 ** (-3.0 * np.repeat(steps, B))
    out["by_element"] = noise * np.repeat(10.0 ** rng.uniform(-30, 30, n // B), B)
    out["by_dof"] = noise * 10.0 ** rng.uniform(-30, 30, n)
    out["bubbles"] = noise * np.where(np.tile(inner, n // B), 1.0, 1e-9)
    out["sparse"] = np.where(np.repeat(rng.random(n // B) < 0.2, B), noise, 0.0)
    return out


@pytest.mark.parametrize("contrast", [1.0, 1e-4])
@pytest.mark.parametrize("kind", sorted(WORKLOADS))
def test_rows_for_vectors_of_any_range(kind, contrast):
    """Values of a neighbour that a row does not see take nothing from it. Beyond
    the bound above a row may lose, of each block, 16 products' low halves: 2^-58 of
    sqrt(A_ii A_jj) times the element's largest |x_j|, which is at most 2^8 times
    the largest one that the row sees: 2^-45 sum_j sqrt(A_ii A_jj) |x_j| over
    the row's entries with room for the roundings to powers of two."""
    from paper_2602_16312_gb300 import aggmg
    wl = WORKLOADS[kind]()
    mesh = _mesh(wl, contrast)
    hier = aggmg.Hierarchy(mesh, 1.0 / wl.dt, wl.maps, precision="f64")
    ref = Rows(mesh, 1.0 / wl.dt)
    d = np.zeros(ref.shape)
    for k in np.nonzero(ref.rows == ref.cols)[0]:
        d[ref.rows[k]] = np.sqrt(np.diag(ref.A[k]).astype(float))
    seen = (ref.A != 0).astype(float)
    for name, x in _vectors(wl, np.random.default_rng(5)).items():
        y, size = ref.product(x)
        part = np.zeros(ref.shape)
        np.add.at(part, ref.rows, (seen * (d * np.abs(x.reshape(ref.shape)))[ref.cols][:, None, :]).sum(2))
        tol = (ref.terms + 8) * 2.0 ** -53 * size + 2.0 ** -45 * (d * part).ravel()
        for level in (0, -1):
            off = np.abs(_apply(hier, x, level) - y)
            worst = int(np.argmax(np.where(tol > 0, off / np.where(tol > 0, tol, 1), 0)))
            assert (off <= tol).all(), (name, level, worst, float(off[worst]), float(size[worst]), float(tol[worst]))
    hier.close()


@pytest.mark.parametrize("skew", [1e-11, 1e-12])
@pytest.mark.parametrize("kind", sorted(WORKLOADS))
def test_rows_with_a_slightly_unsymmetric_conductivity(kind, skew):
    """D_01 = D_10 + skew sqrt(D_00 D_11): the operator's entries and not the means
    of (i, j) and (j, i) are multiplied. The bound takes what the symmetric form may
    differ by where it is kept (7.2e-15 of sqrt(A_ii A_jj))."""
    from paper_2602_16312_gb300 import aggmg
    wl = WORKLOADS[kind]()
    D = wl.conductivity.copy()
    D[:, 0, 1] += skew * np.sqrt(D[:, 0, 0] * D[:, 1, 1])
    mesh = aggmg.Mesh.from_workload(wl, conductivity=D)
    c = 1.0 / wl.dt
    hier = aggmg.Hierarchy(mesh, c, wl.maps, precision="f64")
    ref = Rows(mesh, c)
    d = np.zeros(ref.shape)
    for k in np.nonzero(ref.rows == ref.cols)[0]:
        d[ref.rows[k]] = np.sqrt(np.diag(ref.A[k]).astype(float))
    x = np.random.default_rng(2).standard_normal(wl.n_dofs)
    y, size = ref.product(x)
    root = np.zeros(ref.shape)
    # rms of a sum of random signs: the skew of every entry is bounded on its own
    np.add.at(root, ref.rows, ((ref.A != 0) * (d * x.reshape(ref.shape))[ref.cols][:, None, :].astype(float) ** 2).sum(2))
    tol = (ref.terms + 8) * 2.0 ** -53 * size + 7.2e-15 * (d * np.sqrt(root)).ravel()
    for level in (0, -1):
        off = np.abs(_apply(hier, x, level) - y)
        assert (off <= tol).all(), (level, float((off / tol).max()))
    hier.close()
