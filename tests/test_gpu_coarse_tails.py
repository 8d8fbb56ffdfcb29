"""The coarse-level sums whose loads go in groups (children of a unit, rows of
the coarsest products) at counts around a group: bit for bit the sums of the
persistent kernel, which adds the same terms one by one in the same order."""
import numpy as np
import pytest

from paper_2602_16312_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# elements per side, degree, elements per level-1 unit, level-1 units per level-2 unit:
# 1, 15 .. 17, 33 children; 4, 162, 315, 513, 522 and 648 DoFs on the coarsest level
CASES = [(48, 2, 16, 2), (48, 2, 17, 8), (48, 2, 2, 20), (48, 2, 33, 2), (19, 1, 1, 361), (30, 2, 3, 17),
         (19, 2, 15, 1), (57, 2, 3, 19)]


@pytest.mark.parametrize("form", ["f64", "f32"])
@pytest.mark.parametrize("n,p,g1,g2", CASES)
def test_group_tails_are_bitwise_the_plain_sums(n, p, g1, g2, form):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import aggmg, build
    build.build()
    wl = W.jittered_square_2d(n=n, degree=p, n_levels=2)
    n1 = -(-n * n // g1)
    maps = [np.arange(n * n) // g1, np.arange(n1) // g2]
    mesh = aggmg.Mesh.from_workload(wl)
    r = torch.tensor(np.random.default_rng(7).standard_normal(wl.n_dofs), device="cuda")
    z = []
    for persistent in (False, True):
        h = aggmg.Hierarchy(mesh, 1.0 / wl.dt, maps, precision=form, fine="bsr" if form == "f64" else "mf",
                            coarse_persistent=persistent)
        assert h.launches()["persistent"] == persistent
        z.append(torch.empty_like(r))
        h.vcycle_apply(r, z[-1])
        torch.cuda.synchronize()
        h.close()
    assert torch.isfinite(z[0]).all()
    assert torch.equal(z[0], z[1])
