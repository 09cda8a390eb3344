"""FP64 general kernels with and without per-mode weight tables: 2D plans read tables, 3D plans evaluate
the weights. Both against the CPU oracle at lengths whose axes the general kernels run (lengths without a two-step
plan, periodic axes, the recurrence), with the other step tests' FP64 tolerance (1e-12 over at most four steps)."""
import numpy as np
import pytest

from oracle import etd as oetd
from paper_2209_11922_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# last axis general: 2D with tables; 3D without. Long first axes keep the pencils too many for dense products.
CASES = [((512, 512), "periodic"), ((2048, 96), "periodic"), ((16, 2048), "periodic"), ((1024, 256), "periodic"),
         ((768, 24), "dirichlet"), ((8, 2048), "dirichlet"), ((24, 1536), "dirichlet"),
         ((64, 48, 256), "periodic"), ((96, 48, 96), "periodic"), ((32, 128, 128), "periodic"), ((8, 16, 2048), "dirichlet"),
         ((64, 64, 64), "dirichlet")]


@pytest.mark.parametrize("N,bc", CASES, ids=lambda v: v if isinstance(v, str) else "x".join(map(str, v)))
@pytest.mark.parametrize("scheme", [1, 2])
def test_general_fp64_kernels(N, bc, scheme):
    from paper_2209_11922_gb300.etd import Plan
    U = inputs.uniform_field(inputs.field_shape(N, bc), -0.9, 0.9, 83)
    D, tau, steps = 1e-2, 2e-3, 2
    ref = oetd.run(U, N, tuple(1.0 / n for n in N), D, tau, steps, scheme, bc=bc)
    with Plan(N, D, tau, scheme=scheme, dtype="f64", bc=bc) as pl:
        d = torch.from_numpy(np.ascontiguousarray(U)).cuda()
        pl.run(d, steps)
        got = d.cpu().numpy()
    assert np.linalg.norm(got - ref) <= 1e-12 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
