"""agg_operator_apply_static beside calls that work in the hierarchy's own
buffers, on two streams that nothing orders: each result has the bits of the
same call made alone (level 0 with 16, 27 and 64 DoFs per element, whose float64
product makes a fixed-point copy of x, and 9, whose product does not)."""
import numpy as np
import pytest

from paper_2602_16312_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

WORKLOADS = {
    "quad_q2": lambda: W.jittered_square_2d(n=160, degree=2, n_levels=3),
    "quad_q3": lambda: W.jittered_square_2d(n=120, degree=3, n_levels=3),
    "hex_q2": lambda: W.jittered_cube_3d(n=20, degree=2, n_levels=4, group=2),
    "hex_q3": lambda: W.cube_3d_adjoint(n=10, degree=3, n_levels=3, n_sensors=1),
}


@pytest.mark.parametrize("other", ["level0", "vcycle_level0", "profile"])
@pytest.mark.parametrize("kind", sorted(WORKLOADS))
def test_static_product_beside_the_hierarchys_own_calls(kind, other):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import aggmg, build
    build.build()
    wl = WORKLOADS[kind]()
    hier = aggmg.Hierarchy(aggmg.Mesh.from_workload(wl), 1.0 / wl.dt, wl.maps, precision="f64")
    xa, xb = (torch.tensor(np.random.default_rng(s).standard_normal(wl.n_dofs), device="cuda") for s in (1, 2))
    level = -1 if other == "vcycle_level0" else 0
    ref_a, ref_b = torch.empty_like(xa), torch.empty_like(xb)
    hier.operator_apply(level, xa, ref_a)
    hier.operator_apply_static(0, xb, ref_b)
    torch.cuda.synchronize()
    reps = 30
    ya = [torch.empty_like(xa) for _ in range(reps)]
    yb = [torch.empty_like(xb) for _ in range(reps)]
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    for k in range(reps):
        if other == "profile":
            hier.profile_kernel(0, 1, stream=sa)
        else:
            hier.operator_apply(level, xa, ya[k], stream=sa)
        hier.operator_apply_static(0, xb, yb[k], stream=sb)
    torch.cuda.synchronize()
    for k in range(reps):
        assert torch.equal(yb[k], ref_b), k
        if other != "profile":
            assert torch.equal(ya[k], ref_a), k
    hier.close()


@pytest.mark.parametrize("kind", ["quad_q3", "hex_q2", "hex_q3"])
def test_static_product_equals_the_ordinary_one(kind):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import aggmg, build
    build.build()
    wl = WORKLOADS[kind]()
    hier = aggmg.Hierarchy(aggmg.Mesh.from_workload(wl), 1.0 / wl.dt, wl.maps, precision="f64")
    for seed in range(2):
        x = torch.tensor(np.random.default_rng(seed).standard_normal(wl.n_dofs), device="cuda")
        y, z = torch.empty_like(x), torch.full_like(x, float("nan"))
        hier.operator_apply(0, x, y)
        hier.operator_apply_static(0, x, z)
        torch.cuda.synchronize()
        assert torch.equal(y, z)
    hier.close()
