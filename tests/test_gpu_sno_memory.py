"""Device memory of an operator, and inference where the layers' contractions are wider than a field (n < padded modes)."""
import numpy as np
import pytest

from oracle import sno as osno
from paper_2209_11922_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_creation_holds_no_field_twice():
    """The buffers that training needs (h_0..h_L, z, dh twice, modes, parameters, scratch) and at most 32 MB beside them (the
    allocator's granularity): inference works in buffers of the gradient."""
    from paper_2209_11922_gb300.sno import Sno
    N, C, M, L, B = 256, 32, 24, 2, 64
    n = N - 1
    torch.cuda.init()
    Sno(16, 16, 4, 1, 1).close()   # the library's own start-up
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s = Sno(N, C, M, L, B)
    used = before - torch.cuda.mem_get_info()[0]
    s.close()
    field, modes = B * C * n * n, B * C * M * M
    params = 3 * C + L * (M * M * C * C + C * C + C) + C + 1
    floats = (2 * L + 3) * field + (L + 2) * modes + B * C * n * M + 2 * B * n * n + 4 * params + max(B * C * 16, B * 16 * C * C)
    assert used <= 4 * floats + (32 << 20), (used, 4 * floats)


@pytest.mark.parametrize("N,C,M", [(8, 16, 7), (16, 32, 12), (16, 16, 15), (24, 32, 23)])
def test_inference_with_fewer_rows_than_padded_modes(N, C, M):
    from paper_2209_11922_gb300.sno import Sno
    w = inputs.SnoWorkload("memory", N=N, C=C, M=M, L=2, window=5, tau=1e-2)
    P = w.init_weights()
    P["Wq"] = P["Wq"] * 10
    u = np.stack([w.u0(i) for i in range(3)]).astype(np.float32)
    D = [w.D(i) for i in range(3)]
    OP = osno.Params(*[np.asarray(P[k], dtype=np.float32).astype(np.float64) for k in osno.Params.NAMES])
    ref, _ = osno.forward(OP, u.astype(np.float64), D, N)
    s = Sno(N, C, M, 2, 3)
    s.set_params(P)
    got = s.forward(torch.from_numpy(u).cuda(), D).cpu().numpy()
    s.close()
    assert np.linalg.norm((got - u) - (ref - u)) <= 2e-4 * np.linalg.norm(ref - u)   # the bound of the operator's other forward tests
