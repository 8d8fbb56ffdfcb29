"""agg_kernel_cost of the symmetric level-0 blocks against counts made here from the
mesh: each coupling once, a neighbour id, a block id and a face code per face,
and in float64 the fixed-point copies (8 bytes per DoF, 4 per element) and the scale
exponents (2 bytes per DoF)."""
import pytest

from paper_2602_16312_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _hier(wl, precision, fine):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import aggmg, build
    build.build()
    return aggmg.Hierarchy(aggmg.Mesh.from_workload(wl), 1.0 / wl.dt, wl.maps, precision=precision, fine=fine)


def _counts(n, dim, p):
    """(elements, DoFs, stored entries, entries of the operator, bytes of ids) of n^dim elements."""
    N, E = p + 1, n ** dim
    B, NF = N ** dim, N ** (dim - 1)
    faces = dim * n ** (dim - 1) * (n - 1)
    block = 2 * NF * B - NF * NF
    return E, E * B, E * B * (B + 1) // 2 + faces * block, E * B * B + 2 * faces * block, E * 2 * dim * 9


@pytest.mark.parametrize("kind,n,p", [("jsquare", 12, 3), ("jcube", 5, 2), ("jcube", 3, 3)])
def test_float64_product(kind, n, p):
    dim = 2 if kind == "jsquare" else 3
    wl = W.jittered_square_2d(n=n, degree=p, n_levels=2) if dim == 2 else W.jittered_cube_3d(n=n, degree=p, n_levels=2, group=2)
    hier = _hier(wl, "f32", "mf")
    E, N, stored, entries, ids = _counts(n, dim, p)
    copy = 8 * N + 4 * E
    # x, y; the copy written and read; the scales read by both launches
    assert hier.kernel_cost(0) == (8 * stored + ids + 2 * 8 * N + 2 * copy + 2 * 2 * N, 2 * entries)
    hier.close()


def test_smoothing_step_float32_blocks():
    wl = W.jittered_square_2d(n=20, degree=2, n_levels=2)
    hier = _hier(wl, "f32", "bsr")
    E, N, stored, entries, ids = _counts(20, 2, 2)
    # block inverses as triangles; x, rhs, d in, d and x out
    assert hier.kernel_cost(1) == (4 * stored + ids + 4 * E * 45 + 5 * 4 * N, 2 * entries + 2 * E * 81 + 4 * N)
    hier.close()


def test_smoothing_step_and_iteration_float64_blocks():
    wl = W.jittered_cube_3d(n=5, degree=2, n_levels=2, group=2)
    hier = _hier(wl, "f64", "bsr")
    E, N, stored, entries, ids = _counts(5, 3, 2)
    copy = 8 * N + 4 * E
    step = 8 * stored + ids + 2 * N + 8 * E * 378 + 2 * N + 2 * E + 5 * 8 * N + 2 * copy
    assert hier.kernel_cost(1) == (step, 2 * entries + 2 * E * 729 + 4 * N)
    c = [hier.kernel_cost(k)[0] for k in range(5)]
    # an iteration's product reads p and its copy, which the p update writes: id 0 less
    # one vector; 5 such steps, the restriction and the prolongation besides
    assert c[4] > c[0] - 8 * N + 5 * c[1] - 8 * N + c[2] + c[3]
    assert c[4] < 1.5 * (c[0] + 6 * c[1] + c[2] + c[3]) + 8 * 2 * (hier.stats()["units"][1] * 27) ** 2
    hier.close()
