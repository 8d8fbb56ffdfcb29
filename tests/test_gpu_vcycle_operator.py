"""operator_apply(level=-1) is the operator that the V-cycle's level 0 uses. In
the float64 form with 9 DoFs per element that is the symmetric fixed-point form
(csrc/sym_op.cuh) and level 0, the product of the outer CG, the face-structured
one: the same operator, rounded differently. With 16 and more DoFs both are the
symmetric form, with 4 both the face-structured one, bit for bit.

Tolerance: both sides round a sum of at most 304 products, so 304 * 2^-53 =
3.4e-14 of max |y| (elements of one mesh size); 1e-13 is used."""
import numpy as np
import pytest

from paper_2602_16312_gb300 import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,p,same", [(120, 2, False), (61, 2, False), (40, 3, True), (30, 1, True)])
def test_level_minus_one_is_the_vcycles_operator(n, p, same):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_16312_gb300 import aggmg, build
    build.build()
    wl = W.jittered_square_2d(n=n, degree=p, n_levels=3)
    hier = aggmg.Hierarchy(aggmg.Mesh.from_workload(wl), 1.0 / wl.dt, wl.maps, precision="f64")
    x = torch.tensor(np.random.default_rng(3).standard_normal(wl.n_dofs), device="cuda")
    y0, y1 = torch.empty_like(x), torch.empty_like(x)
    hier.operator_apply(0, x, y0)
    hier.operator_apply(-1, x, y1)
    torch.cuda.synchronize()
    assert float((y1 - y0).abs().max() / y0.abs().max()) <= 1e-13
    assert torch.equal(y0, y1) == same
    hier.close()
